// imrp_field_noalloc: the field evaluation of imrp_get_field for callers that
// cannot allocate device memory (see include/imrp.h). All intermediate
// buffers live in one file-scope device array of fixed size; no call allocates
// or frees device memory. The first call on a device also takes one page-locked
// mapped word of host memory for its error flag, which is kept until exit.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <mutex>
#include <vector>

#include "../../include/imrp.h"
#include "imrp_internal.h"

using namespace imrp;

namespace {

constexpr int64_t kMaxN = IMRP_NOALLOC_MAX_N;
constexpr int kMaxL = IMRP_NOALLOC_MAX_L;

constexpr size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Byte layout of the scratch for n particles, degree L, element size es.
struct Layout {
  size_t part, st[6], id, key0, idx0, key1, idx1, sort, agg, pfx, gagg, gbase, tot, totd, gswork, gsticket, eout,
      step, total;
};
constexpr Layout layout(int64_t n, int L, size_t es) {
  Layout o{};
  const int64_t ntiles = (n + 31) / 32;
  const int64_t ngroups = (ntiles + kTilesPerGroup - 1) / kTilesPerGroup;
  const int64_t nc = 2 * int64_t(ncomp(L));
  size_t at = 0;
  o.part = at; at += align256(size_t(n) * 8 * es);  // Part<T> records: 8 elements each
  for (int k = 0; k < 6; ++k) { o.st[k] = at; at += align256(size_t(n) * es); }
  o.id = at; at += align256(size_t(n) * 4);
  o.key0 = at; at += align256(size_t(n) * 4);
  o.idx0 = at; at += align256(size_t(n) * 4);
  o.key1 = at; at += align256(size_t(n) * 4);
  o.idx1 = at; at += align256(size_t(n) * 4);
  o.sort = at; at += align256(sort_scratch_bytes(n));
  o.agg = at; at += align256(size_t(nc * tile_stride(ntiles)) * es);
  o.pfx = at; at += align256(size_t(nc * tile_stride(ntiles)) * es);
  o.gagg = at; at += align256(size_t(nc * ngroups) * 8);
  o.gbase = at; at += align256(size_t(nc * ngroups) * es);
  o.tot = at; at += align256(size_t(nc) * es);
  o.totd = at; at += align256(size_t(nc) * 8);
  o.gswork = at; at += align256(size_t(gs_work_doubles(int(nc))) * 8);
  o.gsticket = at; at += align256(size_t(gs_tickets(int(nc))) * 4);
  o.eout = at; at += align256(size_t(3 * n) * es);
  o.step = at; at += align256(sizeof(StepState));
  o.total = at;
  return o;
}

constexpr size_t kScratchBytes = layout(kMaxN, kMaxL, sizeof(double)).total;

// The scratch: held by every device that loads this library, until exit.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

std::mutex g_mu;
void* g_addr[64] = {nullptr};  // device address of g_scratch, per device
// error flag per device, in page-locked mapped memory (written by the kernels
// only when there is an error; a call reads it after its wait, without a copy)
volatile int* g_err[64] = {nullptr};
int* g_derr[64] = {nullptr};
// The table of per-degree kernels is built when the library is loaded, so
// that no call allocates host memory for it.
std::vector<KernelSet<float>> g_f;
std::vector<KernelSet<double>> g_d;
struct Registry {
  Registry() { register_all(g_f, g_d); }
};
const Registry g_registry;

template <class T> const std::vector<KernelSet<T>>& sets();
template <> const std::vector<KernelSet<float>>& sets<float>() { return g_f; }
template <> const std::vector<KernelSet<double>>& sets<double>() { return g_d; }

constexpr double kPi = 3.14159265358979323846;
constexpr double kE = 1.602176634e-19;
constexpr double kEps0 = 8.8541878128e-12;

// Per-call set-up of what must start at zero or at the given step: the step
// state, the group scan's tickets and the sort's digit totals (the scratch keeps the
// previous call's contents, and another n or degree lays it out differently).
struct NaInit { StepState* st; int64_t step; unsigned* ticket; int nticket; SortState* sort; int ndigit; };

// FP64 [n][3] positions -> particle records, ids 0..n-1, zero velocities, and their radius keys;
// flags positions outside 1 < r < r_out or non-finite. The first block does the set-up too. (As
// kernels of their own the set-up and the keys took 5 of the 86 us of a call for 1000 particles.)
template <class T>
__global__ void __launch_bounds__(256) k_na_load(const double* __restrict__ x, Part<T>* part, uint32_t* key,
                                                 uint32_t* kidx, int64_t n, double r_out, RadiusKey rk, int* err,
                                                 NaInit in) {
  chain_wait();
  if (blockIdx.x == 0) {
    for (int k = threadIdx.x; k < in.nticket; k += 256) in.ticket[k] = 0u;
    for (int k = threadIdx.x; k < in.ndigit; k += 256) in.sort->tot[k] = 0u;
    if (threadIdx.x == 0) {
      in.sort->ticket = 0u;
      in.st->step = in.step;
      in.st->next = in.step;
      in.st->u = 0.0;
      in.st->kick = 0.0;
      in.st->sync = 0;
      in.st->nabs_step = 0;
      in.st->qs_acc = 0.0;
      in.st->nabs_total = 0;
    }
  }
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double a = x[3 * j], b = x[3 * j + 1], c = x[3 * j + 2];
  Part<T> p;
  p.x = T(a); p.y = T(b); p.z = T(c);
  p.vx = T(0); p.vy = T(0); p.vz = T(0);
  p.id = uint32_t(j);
  const double r2 = double(p.x) * double(p.x) + double(p.y) * double(p.y) + double(p.z) * double(p.z);
  if (!(isfinite(a) && isfinite(b) && isfinite(c))) atomicOr(err, kErrNaN);
  else if (!(r2 > 1.0 && r2 < r_out * r_out)) atomicOr(err, kErrRange);
  part[j] = p;
  key[j] = radius_key<T>(p.x, p.y, p.z, rk);
  kidx[j] = uint32_t(j);
}

cudaError_t preload_noalloc_kernels() {
  cudaFuncAttributes fa;
  const void* fns[] = {reinterpret_cast<const void*>(&k_na_load<float>),
                       reinterpret_cast<const void*>(&k_na_load<double>)};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <class T>
int run(const imrp_params* p, const double* x, int64_t n, int64_t step, double* E, cudaStream_t s,
        unsigned char* base) {
  const int L = p->l_max;
  const KernelSet<T>* ks = nullptr;
  for (const auto& k : sets<T>())
    if (k.L == L) ks = &k;
  if (!ks) return IMRP_E_INVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return IMRP_E_CUDA;
  if (ks->init(dev) != 0) return IMRP_E_CUDA;
  const Layout o = layout(n, L, sizeof(T));
  const double R = p->R_D_m;
  const double d = 1.0 - p->R_E_m / R;
  const double r_out = p->R_out_m / R;
  const double n_tilde = double(n) / (4.0 * kPi / 3.0 * (r_out * r_out * r_out - 1.0));
  const int64_t ntiles = (n + 31) / 32;
  const int64_t ngroups = (ntiles + kTilesPerGroup - 1) / kTilesPerGroup;
  const int nc = 2 * ncomp(L);
  auto P = [&](size_t off) { return static_cast<void*>(base + off); };
  Part<T>* st0 = static_cast<Part<T>*>(P(o.part));
  T* st1[6];
  for (int k = 0; k < 6; ++k) st1[k] = static_cast<T*>(P(o.st[k]));
  uint32_t* id1 = static_cast<uint32_t*>(P(o.id));
  uint32_t* key0 = static_cast<uint32_t*>(P(o.key0));
  uint32_t* idx0 = static_cast<uint32_t*>(P(o.idx0));
  StepState* st = static_cast<StepState*>(P(o.step));
  int* err = g_derr[dev];
  *g_err[dev] = 0;
  LaunchSeq seq(s);
  const NaInit init{st, step, static_cast<unsigned*>(P(o.gsticket)), gs_tickets(nc), static_cast<SortState*>(P(o.sort)),
                    sort_digits(n)};
  seq(k_na_load<T>, unsigned((n + 255) / 256), 256, 0, x, st0, key0, idx0, n, r_out, make_radius_key(r_out), err, init);
  const uint32_t* perm =
      launch_radix_sort<T>(key0, idx0, static_cast<uint32_t*>(P(o.key1)), static_cast<uint32_t*>(P(o.idx1)), P(o.sort),
                           n, sort_first_byte(sizeof(T) == 4 ? 1 : 0), st0, st1, id1, err, seq);
  if (perm) launch_reorder<T>(st0, st1, id1, perm, n, seq);
  MomArgs<T> ma;
  memset(&ma, 0, sizeof(ma));  // all electrons (species = 0)
  ma.x = st1[0]; ma.y = st1[1]; ma.z = st1[2];
  ma.n = n;
  ma.rho = T(r_out);
  ma.rho_inv = T(1.0 / r_out);
  ma.agg = static_cast<T*>(P(o.agg));
  ma.parts = mom_parts(sizeof(T), L, n, mom_ppt(sizeof(T), n));
  ks->moments(ma, seq);
  double canti[kTabL] = {0}, f[kTabL] = {0};
  for (int l = 1; l <= L; ++l) {
    f[l] = coef_f(l, d, p->eps_D);
    canti[l] = coef_canti(l, d, p->eps_D);
  }
  FinalizeArgs fa;
  memset(&fa, 0, sizeof(fa));
  fa.st = st;
  fa.totd = static_cast<const double*>(P(o.totd));
  fa.record = 0;
  fa.L = L;
  fa.drive_kind = p->drive_kind;
  fa.inv_ntilde = 1.0 / n_tilde;
  fa.v_hat = p->V_volts * kEps0 / (p->n_e_m3 * kE * R * R);
  fa.sigma = p->width_wpe;
  fa.t0 = p->t0_wpe > 0 ? p->t0_wpe : 4.0 * p->width_wpe;
  fa.dt = p->dt;
  fa.q_s = p->q_s;
  for (int l = 0; l < kTabL; ++l) {
    fa.canti[l] = canti[l];
    fa.cdrive[l] = canti[l] * 4.0 * kPi * n_tilde;
  }
  launch_scans<T>(static_cast<T*>(P(o.agg)), static_cast<T*>(P(o.pfx)), static_cast<double*>(P(o.gagg)),
                  static_cast<double*>(P(o.gswork)), static_cast<unsigned*>(P(o.gsticket)),
                  static_cast<T*>(P(o.gbase)), static_cast<T*>(P(o.tot)), static_cast<double*>(P(o.totd)), ntiles, nc,
                  32, &fa, seq);
  FieldArgs<T> a;
  memset(&a, 0, sizeof(a));
  a.x = st1[0]; a.y = st1[1]; a.z = st1[2]; a.vx = st1[3]; a.vy = st1[4]; a.vz = st1[5];
  a.id = id1;
  a.key = key0;
  a.kidx = idx0;
  a.n = n;
  a.pfx = static_cast<const T*>(P(o.pfx));
  a.gbase = static_cast<const T*>(P(o.gbase));
  a.tot = static_cast<const T*>(P(o.tot));
  a.agg = static_cast<const T*>(P(o.agg));
  a.img_in_tile = img_in_tile_for<T>(n);
  a.st = st;
  a.Eout = static_cast<T*>(P(o.eout));
  a.err = err;
  a.mode = 1;
  a.L = L;
  a.rho = T(r_out);
  a.rho_inv = T(1.0 / r_out);
  a.pf = 1.0 / (4.0 * kPi * n_tilde);
  a.ion_coef = double(n) / (r_out * r_out * r_out - 1.0);
  a.q_s = p->q_s;
  a.r_out2 = r_out * r_out;
  a.rk = make_radius_key(r_out);
  a.dt = T(p->dt);
  a.r_out = T(r_out);
  a.wall_rule = p->wall_rule;
  a.nabs = nullptr;  // field only: nothing is pushed or absorbed
  a.sigma_v = 0.0;
  a.self_image = p->self_image;
  a.seed = p->seed;
  double rl = 1.0;
  for (int l = 0; l < kTabL; ++l) {
    a.f[l] = T(f[l]);
    a.rhol[l] = T(rl);
    rl *= r_out;
    a.cdrive[l] = canti[l] * 4.0 * kPi * n_tilde;
  }
  derive_field_args(a);
  ks->field(a, 1, seq);  // at most 512 tiles: one per CTA spreads them over the SMs
  const T* eo = static_cast<const T*>(P(o.eout));
  const T* cs[3] = {eo, eo + n, eo + 2 * n};
  launch_scatter_by_id<T>(cs, 3, id1, E, n, seq);
  if (cudaGetLastError() != cudaSuccess) return IMRP_E_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return IMRP_E_CUDA;
  const int h = *g_err[dev];
  if (h & kErrSort) return IMRP_E_CUDA;
  if (h & kErrNaN) return IMRP_E_NAN;
  if (h & kErrRange) return IMRP_E_INVAL;
  return IMRP_OK;
}

}  // namespace

extern "C" int imrp_field_noalloc(const imrp_params* p, const double* x_dev, int64_t n, int64_t step,
                                  double* E_dev, void* stream) {
  if (!p || !x_dev || !E_dev) return IMRP_E_INVAL;
  if (n < 1 || n > kMaxN) return IMRP_E_INVAL;
  if (p->l_max < 1 || p->l_max > kMaxL || p->m0_only != 0) return IMRP_E_INVAL;
  if (p->precision != 0 && p->precision != 1) return IMRP_E_INVAL;
  if (!(p->R_D_m > 0 && p->R_E_m > 0 && p->R_E_m < p->R_D_m && p->R_out_m > p->R_D_m)) return IMRP_E_INVAL;
  if (!(p->eps_D >= 1.0) || !(p->n_e_m3 > 0) || !(p->dt > 0)) return IMRP_E_INVAL;
  if (p->drive_kind < 0 || p->drive_kind > 2 || (p->drive_kind == 0 && !(p->width_wpe > 0))) return IMRP_E_INVAL;
  if (step < 0) return IMRP_E_INVAL;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return IMRP_E_CUDA;
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> g(g_mu);
    if (!g_addr[dev]) {
      // Set-up, once per device: CUDA loads device code lazily, and loading a
      // module reserves device memory (its code and its static arrays, this
      // file's scratch included). So every kernel that a call may launch, in
      // both precisions and at every degree up to the limit, is loaded here,
      // with its tables filled, and later calls load nothing.
      if (preload_core_kernels() != cudaSuccess || preload_noalloc_kernels() != cudaSuccess)
        return IMRP_E_CUDA;
      for (const auto& k : g_f)
        if (k.L <= kMaxL && k.init(dev) != 0) return IMRP_E_CUDA;
      for (const auto& k : g_d)
        if (k.L <= kMaxL && k.init(dev) != 0) return IMRP_E_CUDA;
      void* ptr = nullptr;
      if (cudaGetSymbolAddress(&ptr, g_scratch) != cudaSuccess || !ptr) return IMRP_E_CUDA;
      int *he = nullptr, *de = nullptr;
      if (cudaHostAlloc(&he, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess)
        return IMRP_E_CUDA;
      if (cudaHostGetDevicePointer(&de, he, 0) != cudaSuccess) {
        cudaFreeHost(he);
        return IMRP_E_CUDA;
      }
      g_err[dev] = he;
      g_derr[dev] = de;
      g_addr[dev] = ptr;
    }
    base = static_cast<unsigned char*>(g_addr[dev]);
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return p->precision == 1 ? run<float>(p, x_dev, n, step, E_dev, s, base)
                           : run<double>(p, x_dev, n, step, E_dev, s, base);
}
