// Internal interfaces between the host API (imrp_api.cu), the generic kernels
// (imrp_core.cu) and the per-degree instantiation units (imrp_inst_*.cu).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <atomic>
#include <vector>

#include "imrp_device.cuh"

namespace imrp {

// ---- coefficients (host; written from App. A and Sec. 3 with R = 1) ---------
// f_l of the radial Green's function R^(p,p)_l (App. A).
inline double coef_f(int l, double d, double eps) {
  const double x = pow(1.0 - d, 2 * l + 1);
  return (l * (eps - 1.0) + (l + eps + l * eps) * x) / ((l + 1 + l * eps) + (l + 1) * (eps - 1.0) * x);
}
// b^P_l of the characteristic function outside the dielectric (Sec. 3).
inline double coef_bP(int l, double d, double eps) {
  const double den = (l + 1) * (eps - 1.0) * pow(1.0 - d, 2 * l + 1) + l * eps + l + 1;
  return (2 * l + 1) * eps * pow(1.0 - d, l + 1) / den;
}
// c_l' of Sec. 3 for odd degree l = 2l'-1: (-1/2)^{l'+1} (4l'-1) (2l'-3)!! / l'!
inline double coef_cprime(int lp) {
  double df = 1.0;
  for (int k = 2 * lp - 3; k > 1; k -= 2) df *= k;
  double fact = 1.0;
  for (int k = 2; k <= lp; ++k) fact *= k;
  const double sgn = ((lp + 1) % 2 == 0) ? 1.0 : -1.0;
  return sgn * pow(0.5, lp + 1) * (4.0 * lp - 1.0) * df / fact;
}
// Coefficient of r^{-(l+1)} P_l(cos t) in Psi_anti for r >= R (Sec. 3): c_l' b^P_l
// for odd l = 2l'-1, zero for even l.
inline double coef_canti(int l, double d, double eps) {
  return (l % 2 == 1) ? coef_cprime((l + 1) / 2) * coef_bP(l, d, eps) : 0.0;
}

// Copies host memory to device memory that kernels on any stream may read: the data is there when
// this returns. A plain cudaMemcpy of pageable memory may return before its last transfer to the
// device, and non-blocking streams do not wait for the legacy stream that it runs on.
inline cudaError_t upload(void* dst, const void* src, size_t bytes) {
  const cudaError_t e = cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice);
  return e != cudaSuccess ? e : cudaStreamSynchronize(cudaStreamLegacy);
}

// ---- launches ---------------------------------------------------------------
// A sequence of dependent kernel launches on one stream. A launch whose
// predecessor on the stream is a kernel of the same sequence gets the
// programmatic serialisation attribute (all these kernels begin with
// chain_wait); the first one, and the first after an event or another
// operation (unchain), a full dependency. Step, full dependencies -> chained (us,
// captured graphs): N = 3001, l_max 8: 53.4 -> 51.4; N = 1e5, l_max 16: 97.5 ->
// 94.8; N = 3e5, l_max 8: 108.2 -> 105.0.
struct LaunchSeq {
  cudaStream_t s;
  bool chained = false;
  explicit LaunchSeq(cudaStream_t stream) : s(stream) {}
  void unchain() { chained = false; }
  template <class... P, class... A>
  void operator()(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);  // errors: cudaGetLastError of the caller
    chained = true;
  }
};

// ---- radix sort (imrp_core.cu) ---------------------------------------------
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;  // keys per CTA
constexpr int64_t sort_blocks(int64_t n) { return (n + kSortTile - 1) / kSortTile; }
// Scratch of the bucket sort's first pass: the digits' totals and the ticket of its CTAs, zero
// between sorts (zeroed before the first, in the order of its stream), and the digits' cursors. Behind it stand, for the global
// passes, the block counts of 256 digits per block and the digit totals.
constexpr int kSortDigits = 8192;
struct alignas(64) SortState {
  uint32_t tot[kSortDigits], cur[kSortDigits], ticket;
};
constexpr size_t sort_scratch_bytes(int64_t n) {
  return sizeof(SortState) + sizeof(uint32_t) * size_t(256 * sort_blocks(n) + 256);
}
int sort_digits(int64_t n);  // digits of the first pass for n keys alone on the GPU
// Sorts the particles src[0 .. n) by the key bytes first_byte..3 (stable: keys equal in those
// bytes keep their order). k0/v0 hold the keys and slots 0 .. n-1; k1/v1 are scratch of n;
// scratch: sort_scratch_bytes(n). Either gathers the particles into the component arrays dst and
// id_dst itself and returns null, or returns the buffer that holds the slots in key order. err
// receives kErrSort if the sort state was not in order (then the order is not to be used).
// Key bytes sorted: all four, in both precisions. The radius key is
// floor((r^2 - 1) / (r_out^2 - 1) * 2^32) of the exact FP64 r^2 of the stored
// position, and the sorted index j of a particle is its count of electrons
// inside (the l = 0 term), which jumps by one electron per misordered pair;
// so even radii that FP32 arithmetic cannot tell apart are ordered exactly.
inline int sort_first_byte(int) { return 0; }
template <class T>
const uint32_t* launch_radix_sort(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, void* scratch, int64_t n,
                                  int first_byte, const Part<T>* src, T* const* dst, uint32_t* id_dst, int* err,
                                  LaunchSeq& seq, bool shared_gpu = false);

// ---- state movement and keys (imrp_core.cu) ---------------------------------
// The state is an array of Part<T> records in the order of the last push (or
// load); each step gathers it into radius order as component arrays.
template <class T>
void launch_reorder(const Part<T>* src, T* const* dst, uint32_t* id_dst, const uint32_t* perm, int64_t n,
                    LaunchSeq& seq);
template <class T>
void launch_keys(const Part<T>* st, uint32_t* key, uint32_t* kidx, int64_t n, double r_out, LaunchSeq& seq);
template <class T>
void launch_load(const double* x /* [n][3] */, const double* v /* [n][3] */, const uint32_t* ids /* or null */,
                 Part<T>* st, uint32_t* key, uint32_t* kidx, int64_t n, double r_out, int* err, cudaStream_t s);
// The state in its storage order: x[j][3], v[j][3], id[j] (checkpoint).
template <class T>
void launch_state_dump(const Part<T>* st, double* x, double* v, uint32_t* id, int64_t n, cudaStream_t s);
// out[id[j]][c] = comp_c[j] for c < ncomp
template <class T>
void launch_scatter_by_id(const T* const* comps, int ncomp, const uint32_t* id, double* out,
                          int64_t n, LaunchSeq& seq);
// the state in id order: x[n][3], v[n][3] (FP64); inv: scratch of n words
template <class T>
void launch_state_out(const Part<T>* st, double* x, double* v, uint32_t* inv, int64_t n, cudaStream_t s);

// ---- scans (imrp_core.cu) ---------------------------------------------------
struct FinalizeArgs {
  StepState* st;
  const double* totd;
  double* qhist;     // qhist[n - first] holds Q_diff of step n (first: step of the load or restore)
  double* uhist;
  int64_t cap;
  int64_t first;
  int record;
  int L;
  int drive_kind;
  double inv_ntilde;
  double v_hat, sigma, t0, dt;
  double canti[kTabL];
  double cdrive[kTabL];  // 4 pi n~ canti (FieldArgs::cdrive)
  double q_s;            // surface charge of the parameters (FieldArgs::q_s)
};
// The derived scalars of a FieldArgs whose pf, rho_inv, r_out2, self_image and
// img_in_tile are set.
template <class T> inline void derive_field_args(FieldArgs<T>& a) {
  a.pf_t = T(a.pf);
  a.mpf = T(-a.pf);
  a.mpfr = T(-a.pf) * a.rho_inv;
  // the image moments include the particle itself, or (img_in_tile) leave its tile out
  a.self_sign = a.img_in_tile ? (a.self_image ? 1 : 0) : (a.self_image ? 0 : -1);
  a.self_pf = T(a.self_sign * a.pf);
  a.near_hi = T(a.r_out2 * (1.0 - 1e-5));
  a.ion_coef_h = float(a.ion_coef);
  a.ion_coef_l = float(a.ion_coef - double(a.ion_coef_h));
}
// In-group scans of agg[u][tile] (row stride tile_stride(ntiles)) into
// pfx[tile][u] (tile-major: one tile's nc carries contiguous), the group totals
// gagg[g][u] (FP64), and the scan over the groups into gbase and the totals tot
// and totd. gseg: least number of groups per segment (16, 32 or 64; chosen by the
// autotuner). work: gs_work_doubles(nc) doubles; ticket: gs_tickets(nc)
// counters, zero before the first call (each call leaves them zero). fin (or
// null): the step's finalize (drive, kick weight, Q_diff tally), run once the
// totals are complete.
template <class T>
void launch_scans(const T* agg, T* pfx, double* gagg, double* work, unsigned* ticket, T* gbase, T* tot, double* totd,
                  int64_t ntiles, int nc, int gseg, const FinalizeArgs* fin, LaunchSeq& seq);
// Loads the device code of the degree-independent kernels of both precisions that
// the allocation-free entry point can launch, and of some others (CUDA loads
// device code lazily, at a kernel's first launch or query, and the load reserves
// device memory): that entry point calls it at its set-up so that its later
// calls load nothing. (The read-back by ids and the transform are not among them.)
cudaError_t preload_core_kernels();
// opt-in shared memory of the sort's bucket kernel (once per device, before
// the first sort)
cudaError_t set_sort_attributes();
void launch_init_step(StepState* st, cudaStream_t s);

// Spectrum sums: Qh[j] = dt sum_n (q_n - q_0) e^{-i w_j t_n},
// Uh[j] = sum_n kw_n u_n e^{-i w_j t_n}, w_j = (j+1) w_max / nf. work:
// dft_work_doubles(ns, nf) doubles, of which the first [nf][4] receive the sums
// (Q re, im, U re, im) and the rest is scratch.
int64_t dft_work_doubles(int64_t ns, int64_t nf);
void launch_dft(const double* q, const double* u, int64_t ns, double dt, double first_kick,
                int64_t nf, double w_max, double* work, cudaStream_t s);

// ---- per-degree kernels (imrp_inst_*.cu) ------------------------------------
// SMs of the current device (cached per device; contexts may be created from
// several host threads, hence the atomics)
inline int sm_count() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  int c = cache[dev].load(std::memory_order_relaxed);
  if (c == 0) {
    int v = 0;
    c = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0 ? v : 152;
    cache[dev].store(c, std::memory_order_relaxed);
  }
  return c;
}
// Particles per thread of the moments kernel for an instance of n particles:
// 16 (1024 per CTA of 64 threads), or 4 (256 per CTA) for an FP64 instance of
// fewer than 100 such blocks, whose columns alone (below) would not fill the
// GPU: FP64 N = 60000, l_max = 12 took 0.184 ms with 4 and 0.219 with 16;
// N = 250001, l_max = 16 (245 blocks) 1.19 and 0.96, since with 4 each tile's
// sums go over 8 threads. FP32 keeps 16 (N = 1e5, l_max = 16: 0.045 -> 0.068 ms
// with 4).
inline int mom_ppt(int elem_size, int64_t n) { return (elem_size == 8 && (n + 1023) / 1024 < 100) ? 4 : 16; }
// CTAs of the moments kernel per column range (64 threads of ppt particles):
// whole scan groups of 1024 particles, so that every tile the scans read is written
inline int64_t mom_blocks(int64_t n, int ppt) { return (n + 1023) / 1024 * (16 / ppt); }
// Column ranges per block of the moments kernel: a small instance has too few
// blocks for the SMs (N = 1e5: 98 CTAs of two warps), so its columns m are cut
// into ranges that separate CTAs take (a range first walks its particles'
// diagonal terms up to its first column). As many ranges as give the stated
// CTAs per SM: FP32 N = 1e5, l_max = 16: 0.043 ms with one range, 0.0225 with
// 6 per SM, 0.028 with 8; N = 3e5, l_max = 8: 0.0262, 0.0206, 0.0267 (0.0204 and
// 0.0172 since all of a thread's loads go out at once); FP64
// N = 20000, l_max = 8: 0.102 with one, 0.039 with 7 ranges (4 CTAs per SM), 0.043 with 9.
inline int mom_parts(int elem_size, int L, int64_t n, int ppt) {
  const int per_sm = elem_size == 4 ? 6 : ppt == 4 ? 4 : 8;
  const int64_t want = int64_t(per_sm) * sm_count() / mom_blocks(n, ppt);
  return int(want < 1 ? 1 : want > L + 1 ? L + 1 : want);
}

template <class T> struct KernelSet {
  int L;
  void (*moments)(const MomArgs<T>&, LaunchSeq&);
  void (*field)(const FieldArgs<T>&, int wpb, LaunchSeq&);
  int (*init)(int device);  // tables + attributes, once per device
  size_t smem_per_warp;
  int (*field_blocks_per_sm)(int wpb);  // occupancy of the field kernel at wpb warps per CTA
  // Batched launches over several instances of this degree and precision:
  // args[i] in device memory, items[b] = (instance, block) for the moments
  // (item = block parts + column range, ppt = mom_ppt of every listed
  // instance) and (instance, first tile) for the field (CTAs of wpb tiles).
  void (*moments_batch)(const MomArgs<T>* args, const int2* items, int nitems, int ppt, cudaStream_t);
  void (*field_batch)(const FieldArgs<T>* args, const int2* items, int nitems, int wpb, cudaStream_t);
  // the same for instances of field_pair_rule: (instance, first pair of tiles), kPairWarps pairs
  // per CTA; or of field_team_rule: (instance, tile)
  void (*alt_batch)(const FieldArgs<T>* args, const int2* items, int nitems, cudaStream_t);
};
void register_all(std::vector<KernelSet<float>>& f, std::vector<KernelSet<double>>& d);

}  // namespace imrp
