// Per-degree kernel templates of the IMRP hot path: tile moments and the fused
// field gather + leapfrog push + wall + next radius key. Included by the
// instantiation units imrp_inst_*.cu, each of which owns its copy of the
// recurrence tables in constant memory.
#pragma once

#include <type_traits>

#include "imrp_device.cuh"

namespace imrp {

// Recurrence tables of this translation unit (filled by init_tables<T>()).
static __constant__ Tables<float> c_tab_f;
static __constant__ Tables<double> c_tab_d;
template <class T> __device__ __forceinline__ const Tables<T>& tab();
template <> __device__ __forceinline__ const Tables<float>& tab<float>() { return c_tab_f; }
template <> __device__ __forceinline__ const Tables<double>& tab<double>() { return c_tab_d; }

// Per-degree prologue tables of the field kernel, in global memory of this
// translation unit (filled by fill_prologue_tables at initialisation), for
// every instantiated degree.
// EntryRec: one gradient entry k of the shared-memory coefficient arrays.
// Its six sources are scratch entries (the zero slot 2 ncomp(L) where a ladder
// step leaves the table); the factors are the ladder factors times nu of the
// evaluated harmonic, with the 1/2 of d/dx and d/dy, the 2 of the m > 0
// entries and the sign of a negative-m source (X^{-m} = (-1)^m conj(X^m))
// folded in, so the entry is
//   d/dx = s1r c1.re + s2 c2.re + i (s1i c1.im + s2 c2.im)
//   d/dy = (s2 c2.im - s1i c1.im) + i (s1r c1.re - s2 c2.re),  d/dz = sz c0.
struct __align__(16) EntryRec {
  int16_t src[6];   // scratch index of c1.re, c1.im, c2.re, c2.im, c0.re, c0.im
  uint16_t pad[2];
  float s1r, s1i, s2, sz;
};
constexpr int kNumDegrees = 7;  // the instantiated degrees: 1, 2, 4, 8, 12, 16, 24
__host__ __device__ constexpr int degree_at(int i) {
  return i == 0 ? 1 : i == 1 ? 2 : i == 2 ? 4 : i == 3 ? 8 : i == 4 ? 12 : i == 5 ? 16 : 24;
}
__host__ __device__ constexpr int ent_off(int L) {
  int o = 0;
  for (int i = 0; i < kNumDegrees; ++i) {
    const int d = degree_at(i);
    if (d == L) return o;
    o += nI(d) + nR(d);
  }
  return -1;
}
__host__ __device__ constexpr int comp_tab_off(int L) {
  int o = 0;
  for (int i = 0; i < kNumDegrees; ++i) {
    const int d = degree_at(i);
    if (d == L) return o;
    o += ncomp(d);
  }
  return -1;
}
constexpr int kEntTotal = ent_off(24) + nI(24) + nR(24);
constexpr int kCompTotal = comp_tab_off(24) + ncomp(24);
// Recurrence coefficients an_lm of the field's pair kernel, twice each (one
// instruction advances two recurrences), by columns: [m][l - m].
static __constant__ float2 c_an2[kTabL * kTabL];
// Record offP(L, m) + l - m of the pair kernel (columns m, degrees l = m..L + 1): the
// sources (complex coefficients at pair_pos: c1, c2, c0 of the multipole entry (l, m),
// then of the local one) and the factors (s1r, s1i, s2, sz) of the two entries, as in
// EntryRec; factors 0 where a part has no such entry. Arrays of 16-byte parts, so
// that a warp's loads are contiguous.
struct __align__(16) PairSrc { int16_t i[8]; };
__host__ __device__ constexpr int pair_run(int L) { return L + L * (L + 1) / 2; }
__host__ __device__ constexpr int pair_pos(int L, int l, int m, int s) {
  return s * pair_run(L) + (m == 0 ? l - 1 : L + (m - 1) * (L + 1) - (m - 1) * m / 2 + l - m);
}
__host__ __device__ constexpr int nP(int L) { return nI(L) + 1; }
__host__ __device__ constexpr int offP(int L, int m) { return m == 0 ? 0 : offI(L, m) + 1; }
__host__ __device__ constexpr int rec_off(int L) {
  int o = 0;
  for (int i = 0; i < kNumDegrees; ++i) {
    const int d = degree_at(i);
    if (d == L) return o;
    o += nP(d);
  }
  return -1;
}
constexpr int kRecTotal = rec_off(24) + nP(24);
static __device__ PairSrc g_psrc[kRecTotal];
static __device__ float4 g_pfac[2][kRecTotal];  // multipole, local
// the same factors for the FP64 kernel, times the diagonal's constants up to column m. They are the
// EntryRec's, rounded to FP32: that rounding is the FP64 field's error (2.8e-8 at N = 2e6, l_max = 16)
struct __align__(16) TeamFac { double s1r, s1i, s2, sz; };
static __device__ TeamFac g_tfac[2][kRecTotal];
static __device__ EntryRec g_ent[kEntTotal];
static __device__ uint16_t g_comp[kCompTotal];  // per component: l | (drive << 8) | (m > 0) << 9

template <class T> __device__ __forceinline__ T rsqrt_t(T v);
template <> __device__ __forceinline__ float rsqrt_t<float>(float v) { return rsqrtf(v); }
template <> __device__ __forceinline__ double rsqrt_t<double>(double v) { return rsqrt(v); }
template <class T> __device__ __forceinline__ T fma_t(T x, T y, T z);
template <> __device__ __forceinline__ float fma_t<float>(float x, float y, float z) { return fmaf(x, y, z); }
template <> __device__ __forceinline__ double fma_t<double>(double x, double y, double z) { return fma(x, y, z); }

// Tile moments: the sums over each tile of 32 radius-sorted particles of
// q Rs_l^m(x/r_out) and q Is_l^m(x), 1 <= l <= L (q = -1 per electron).
// Two threads per tile, 16 particles each. The recurrences run column by
// column (fixed m, rising l = m + j) in a rolled loop over m, so the code
// stays small at any degree; the column sums stay in registers while the
// thread walks its particles (kMomChains at a time: independent recurrence
// chains), whose scaled positions, r_out / r^2 and diagonal terms live in
// shared memory in a [particle][thread] layout (conflict-free). The multipole
// harmonics follow from the regular ones by the Kelvin relation
//   Is_l^m(x) = Rs_l^m(x / r_out) * r_out^l / r^(2l+1),
// the scale advancing by one factor r_out / r^2 per degree. A CTA of 64
// threads takes 64 PPT particles (2 PPT tiles), PPT particles per thread,
// 32 / PPT threads per tile, and all columns or (small instances, mom_parts)
// one of several ranges of them.
// At the end of a column the threads of each tile are combined: with two
// (PPT = 16), one shuffle per Rs/Is pair (the even lane keeps the Rs sum, the
// odd lane the Is sum); with more, by halving over the tile's threads, each
// then writing its share. Written: agg[u][tile], u = 2 e + s (s = 0 Rs, s = 1 Is).
constexpr int kMomThreads = 64;
constexpr int kMomPPT = 16;       // particles per thread (1024 per CTA) when that fills the GPU
constexpr int kMomPPTSmall = 4;   // particles per thread (256 per CTA) of small FP64 instances (mom_ppt)
constexpr int kMomBreak = 2;      // steps between the column-end tests
// particles advanced together (independent recurrence chains): four in FP32
// (N = 2e6, l_max = 16: 0.174 -> 0.168 ms against two; l_max = 24, N = 4e6:
// 0.676 -> 0.652 ms, though 150 registers lower the occupancy there), two in
// FP64, where four would spill at l_max = 24
template <class T, int L>
__host__ __device__ constexpr int mom_chains() { return sizeof(T) == 4 ? 4 : 2; }

template <class T, int L, int PPT = kMomPPT>
__host__ __device__ constexpr size_t moments_smem() {
  return sizeof(T) * 7 * PPT * (kMomThreads + 1);
}

// First column of part p when the columns m = 0..L are cut into `parts`
// contiguous ranges of about equal work (a column's entries and its fixed cost,
// about two entries' worth).
__device__ __forceinline__ int mom_part_begin(int L, int parts, int p) {
  const int total = (L + 1) * (L + 2) / 2 + 2 * (L + 1);
  const int want = total * p / parts;
  int m = 0, acc = 0;
  while (m <= L && acc < want) acc += L - m++ + 3;
  return m;
}

// (a b.x + c.x, a b.y + c.y): one instruction in FP32, rounded as two. A column's Rs and Is
// sums advance together by it (N = 2e6, l_max = 16: 0.163 -> 0.154 ms; l_max = 24, N = 4e6:
// 0.560 -> 0.539). The FMA pipe's lanes bound the kernel (52 % of its cycles, 12 warps per SM):
// pairing the recurrences too, of Rs and of Is, issues 5 instead of 7 instructions per entry
// and takes 0.156 and 0.542 ms.
template <class T> struct __align__(2 * sizeof(T)) Pair { T x, y; };
__device__ __forceinline__ Pair<float> fma_pair(float a, Pair<float> b, Pair<float> c) {
  const float2 r = __ffma2_rn(make_float2(a, a), make_float2(b.x, b.y), make_float2(c.x, c.y));
  return {r.x, r.y};
}
__device__ __forceinline__ Pair<double> fma_pair(double a, Pair<double> b, Pair<double> c) {
  return {fma(a, b.x, c.x), fma(a, b.y, c.y)};
}

// Diagonal step of the regular harmonics: Rs_m^m = (cx + i cy) Rs_{m-1}^{m-1}. The
// roundings are written out, so that a column range that starts past m = 0 and
// one that walks there have the same diagonal bit for bit.
template <class T> __device__ __forceinline__ void diag_step(T cx, T cy, T& Dr, T& Di) {
  const T nr = fma_t(cx, Dr, -(cy * Di)), ni = fma_t(cy, Dr, cx * Di);
  Dr = nr;
  Di = ni;
}

// Body of the moments kernel for item `item` (block item / parts of the
// instance, column range item % parts) of the instance whose arguments are `a`
// (a kernel parameter, or a copy in shared memory for the batched launch).
template <class T, int L, int PPT>
__device__ __forceinline__ void moments_block(const MomArgs<T>& a, int64_t item, unsigned char* smem_raw) {
  constexpr int NT = kMomThreads;  // threads of the CTA
  constexpr int TPT = 32 / PPT;    // threads per tile
  constexpr int S = NT + 1;       // padded row
  T* sx = reinterpret_cast<T*>(smem_raw);  // x / r_out
  T* sy = sx + PPT * S;                    // y / r_out
  T* sz = sy + PPT * S;                    // z / r_out
  T* sq = sz + PPT * S;                    // r_out / r^2
  T* sRr = sq + PPT * S;                   // q Rs_m^m(x / r_out), real and imaginary
  T* sRi = sRr + PPT * S;
  T* ssc = sRi + PPT * S;                  // r_out^m / r^(2m+1)
  const Tables<T>& tb = tab<T>();
  const int th = threadIdx.x;
  const int64_t ntiles = (a.n + 31) >> 5;
  const int64_t blk = a.parts == 1 ? item : item / a.parts;
  const int part = int(item - blk * a.parts);
  const int mlo = part == 0 ? 0 : mom_part_begin(L, a.parts, part);
  const int mhi = part == a.parts - 1 ? L + 1 : mom_part_begin(L, a.parts, part + 1);
  const int64_t pbase = blk * (NT * PPT);
  const T ri = a.rho_inv;
  constexpr int kMomChains = mom_chains<T, L>() < PPT ? mom_chains<T, L>() : PPT;
  // stage 1024 particles: particle k of the CTA goes to row k % PPT, column k / PPT. A thread's
  // loads are all in flight at once (four particles at a time: N = 5e5, l_max = 1 0.0142 ->
  // 0.0096 ms; N = 3e5, l_max = 8 0.0205 -> 0.0179; N = 2e6, l_max = 16 0.154 -> 0.151)
  T PX[PPT], PY[PPT], PZ[PPT];
  unsigned ions = 0;  // bit i: particle i is a mobile ion
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    const int64_t j = pbase + i * NT + th;
    const bool valid = j < a.n;
    PX[i] = valid ? a.x[j] : T(1); PY[i] = valid ? a.y[j] : T(0); PZ[i] = valid ? a.z[j] : T(0);
  }
  if (a.species) {
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
      const int64_t j = pbase + i * NT + th;
      if (j < a.n && a.id[j] >= a.n_e) ions |= 1u << i;
    }
  }
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    const int k = i * NT + th;
    const int64_t j = pbase + k;
    const bool valid = j < a.n;
    const T X = PX[i], Y = PY[i], Z = PZ[i];
    const int o = (k % PPT) * S + k / PPT;
    const T r2 = fma_t(Z, Z, fma_t(Y, Y, X * X));
    // FP64: from the reciprocal root, which is needed anyway, with one correction by the
    // remainder (a division costs some 20 FP64 operations, and every column range stages its
    // particles). q enters to the power of the degree: without the correction the sums of a
    // particle near the equator are 2.4 times as far off at l_max = 24 as with a division, with it
    // they are as near.
    T ir = rsqrt_t(r2), q;
    if constexpr (sizeof(T) == 8) {
      q = a.rho * (ir * ir);
      q = fma(fma(-q, r2, a.rho), ir * ir, q);
    } else {
      q = a.rho / r2;
    }
    sx[o] = X * ri; sy[o] = Y * ri; sz[o] = Z * ri;
    sq[o] = q;
    // the particle's charge seeds its harmonics: -1 for an electron, q_ion
    // for a mobile ion
    T Dr = valid ? (((ions >> i) & 1u) ? a.q_ion : T(-1)) : T(0), Di = T(0), sc = ir;
    for (int m = 1; m < mlo; ++m) {  // the diagonal up to the column before this part's first
      diag_step(tb.dg[m] * (X * ri), tb.dg[m] * (Y * ri), Dr, Di);
      sc *= q;
    }
    sRr[o] = Dr;
    sRi[o] = Di;
    ssc[o] = sc;
  }
  __syncthreads();
  const int sub = th % TPT;  // this thread's part of its tile
  const bool odd = (th & 1) != 0;
  const int64_t tile = blk * (NT * PPT / 32) + th / TPT;
  if (a.species && part == 0) {
    // the tile's charge (FP64): this thread's particles, then the tile's threads
    double qs = 0.0;
#pragma unroll
    for (int p = 0; p < PPT; ++p) qs += double(sRr[p * S + th]);
#pragma unroll
    for (int d = 1; d < TPT; d <<= 1) qs += __shfl_xor_sync(0xffffffffu, qs, d);
    if (sub == 0) a.qtile[tile] = qs;
  }
  // every tile of the whole groups is written (tiles past the particles hold
  // zeros: their particles carry no charge)
  const int64_t ts = tile_stride(ntiles);
  T* const agg_t = a.agg + tile + (odd ? ts : 0);  // row u = 2 e + odd

#pragma unroll 1
  for (int m = mlo; m < mhi; ++m) {
    Pair<T> acc2[2 * (L + 1)];  // [j][re, im] of (Rs, Is), l = m + j
#pragma unroll
    for (int k = 0; k < 2 * (L + 1); ++k) acc2[k] = Pair<T>{T(0), T(0)};
    T cA[L + 1];  // recurrence coefficients of this column (rescaled harmonics)
#pragma unroll
    for (int j = 1; j <= L; ++j) cA[j] = m + j <= L ? tb.an[(m + j) * kTabL + m] : T(0);
    const T dg = tb.dg[m];
#pragma unroll 1
    for (int p = 0; p < PPT; p += kMomChains) {
      // a column's harmonics are the diagonal Rs_m^m = (Dr + i Di) times a real
      // p_l that obeys the column's three-term recurrence from p_m = 1 (the
      // roundings written out: they don't depend on the code around them)
      T Zs[kMomChains], rs2[kMomChains], q[kMomChains], Dr[kMomChains], Di[kMomChains], P1[kMomChains],
          P0[kMomChains], sc[kMomChains];
#pragma unroll
      for (int u = 0; u < kMomChains; ++u) {
        const int o = (p + u) * S + th;
        const T Xs = sx[o], Ys = sy[o];
        Zs[u] = sz[o]; q[u] = sq[o];
        Dr[u] = sRr[o]; Di[u] = sRi[o]; sc[u] = ssc[o];
        if (m > 0) {  // diagonal step: Rs_m^m = dg_m (x + i y) / r_out * Rs_{m-1}^{m-1}
          diag_step(dg * Xs, dg * Ys, Dr[u], Di[u]);
          sc[u] *= q[u];
          sRr[o] = Dr[u]; sRi[o] = Di[u]; ssc[o] = sc[u];
        }
        rs2[u] = fma_t(Zs[u], Zs[u], fma_t(Xs, Xs, Ys * Ys));
        P1[u] = T(1); P0[u] = T(0);
      }
      if (m > 0) {
#pragma unroll
        for (int u = 0; u < kMomChains; ++u) {
          const Pair<T> v{T(1), sc[u]};
          acc2[0] = fma_pair(Dr[u], v, acc2[0]);
          acc2[1] = fma_pair(Di[u], v, acc2[1]);
        }
      }
#pragma unroll
      for (int j = 1; j <= L; ++j) {
        // the column ends at j = L - m; the test runs every kMomBreak steps (the
        // coefficients past the end are zero, so the extra steps add zeros to
        // sums that are not written)
        if ((j - 1) % kMomBreak == 0 && m + j > L) break;
#pragma unroll
        for (int u = 0; u < kMomChains; ++u) {
          const T az = cA[j] * Zs[u];
          const T pn = fma_t(az, P1[u], -(rs2[u] * P0[u]));
          P0[u] = P1[u]; P1[u] = pn;
          sc[u] *= q[u];
          const Pair<T> v{pn, pn * sc[u]};
          acc2[2 * j] = fma_pair(Dr[u], v, acc2[2 * j]);
          acc2[2 * j + 1] = fma_pair(Di[u], v, acc2[2 * j + 1]);
        }
      }
    }
    // ---- tile sums of the column, pair p = packed component e0 + p
    // (m = 0: p = l - 1, acc(4 l + s); m > 0: p = 2 j + part, acc(2 p + s))
    const int64_t e0 = col_off(L, m);
    const auto acc = [&](int k) { return k % 2 ? acc2[k / 2].y : acc2[k / 2].x; };
    if constexpr (TPT == 2) {
      if (m == 0) {
#pragma unroll
        for (int p = 0; p < L; ++p) {
          const T send = odd ? acc(4 * (p + 1)) : acc(4 * (p + 1) + 1);
          const T recv = __shfl_xor_sync(0xffffffffu, send, 1);
          const T v = (odd ? acc(4 * (p + 1) + 1) : acc(4 * (p + 1))) + recv;
          agg_t[(2 * (e0 + p)) * ts] = v * tb.nu[(p + 1) * kTabL];
        }
      } else {
        const int np = 2 * (L - m + 1);
#pragma unroll
        for (int p = 0; p < 2 * L; ++p) {
          if (p >= np) break;
          const T send = odd ? acc(2 * p) : acc(2 * p + 1);
          const T recv = __shfl_xor_sync(0xffffffffu, send, 1);
          const T v = (odd ? acc(2 * p + 1) : acc(2 * p)) + recv;
          agg_t[(2 * (e0 + p)) * ts] = v * tb.nu[(m + (p >> 1)) * kTabL + m];
        }
      }
    } else {
      // sums over the tile's threads, TPT values at a time by halving (each step a thread
      // keeps half of its values and adds its partner's share of them), so that value k of a
      // run of TPT ends on the thread sub = k
      T* const agg_c = a.agg + tile;
      const int nv = m == 0 ? 2 * L : 4 * (L - m + 1);  // values of the column, (Rs, Is) pairs
      constexpr int NV = 4 * L;
#pragma unroll
      for (int v0 = 0; v0 < NV; v0 += TPT) {
        if (v0 >= nv) break;
        T v[TPT];
#pragma unroll
        for (int k = 0; k < TPT; ++k) {
          // m = 0: value 2 p + s is acc(4 (p + 1) + s) (no imaginary part); else acc(2 p + s)
          const int i0 = 4 * ((v0 + k) / 2 + 1) + (v0 + k) % 2, i1 = v0 + k;
          const T x0 = i0 < 4 * (L + 1) ? acc(i0 < 4 * (L + 1) ? i0 : 0) : T(0);
          v[k] = m == 0 ? x0 : acc(i1);
        }
#pragma unroll
        for (int d = TPT / 2; d >= 1; d >>= 1) {
          const bool up = (sub & d) != 0;
#pragma unroll
          for (int k = 0; k < d; ++k) {
            const T send = up ? v[k] : v[k + d], keep = up ? v[k + d] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, d);
          }
        }
        const int val = v0 + sub;
        if (val < nv) {
          const int l = m == 0 ? val / 2 + 1 : m + val / 4;
          agg_c[(2 * e0 + val) * ts] = v[0] * tb.nu[l * kTabL + m];
        }
      }
    }
  }
}

template <class T, int L, int PPT>
__global__ void __launch_bounds__(kMomThreads) k_moments(MomArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chain_wait();
  moments_block<T, L, PPT>(a, blockIdx.x, smem_raw);
}

// Batched moments: CTA b takes item items[b].y (block and column range) of
// instance items[b].x, whose arguments args[items[b].x] are first copied to
// shared memory.
template <class T> __device__ __forceinline__ void copy_args(const T* src, T* dst) {
  static_assert(sizeof(T) % 4 == 0, "argument blocks are copied in words");
  const uint32_t* s = reinterpret_cast<const uint32_t*>(src);
  uint32_t* d = reinterpret_cast<uint32_t*>(dst);
  for (int k = threadIdx.x; k < int(sizeof(T) / 4); k += blockDim.x) d[k] = s[k];
}
template <class T, int L, int PPT>
__global__ void __launch_bounds__(kMomThreads) k_moments_batch(const MomArgs<T>* __restrict__ args,
                                                               const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ MomArgs<T> sa;
  const int2 it = items[blockIdx.x];
  copy_args(args + it.x, &sa);
  __syncthreads();
  moments_block<T, L, PPT>(sa, it.y, smem_raw);
}

// Constants of the scaled Legendre recurrences of the near field. With
// c_l = (2l-1)!!/l! (the leading coefficient of P_l), q_l = s^l P_l(u) / c_l
// follows q_{l+1} = (s u) q_l - g_l s^2 q_{l-1}, g_l = l^2 / (4 l^2 - 1)
// (Bonnet's recurrence divided by c_{l+1}); and with eps_{l+1} = (2l+1) c_l,
// e_l = s^{l-1} P'_l(u) / eps_l follows e_{l+1} = r_l s^2 e_{l-1} + q_l,
// r_l = eps_{l-1} / eps_{l+1} (from P'_{l+1} = P'_{l-1} + (2l+1) P_l).
__host__ __device__ constexpr double leg_c(int l) {
  double c = 1.0;
  for (int k = 1; k <= l; ++k) c *= double(2 * k - 1) / double(k);
  return c;
}
__host__ __device__ constexpr double leg_g(int l) { return double(l) * l / (4.0 * l * l - 1.0); }
__host__ __device__ constexpr double leg_eps(int l) { return l == 0 ? 1.0 : double(2 * l - 1) * leg_c(l - 1); }
__host__ __device__ constexpr double leg_r(int l) { return leg_eps(l - 1) / leg_eps(l + 1); }

// u_asy(t_n) cdrive[l] and the kick weight of the step, in T.
__device__ __forceinline__ float drive_of(const FieldArgs<float>& a, int l) { return a.st->drive_f[l]; }
__device__ __forceinline__ double drive_of(const FieldArgs<double>& a, int l) { return a.st->u * a.cdrive[l]; }
__device__ __forceinline__ float kick_of(const FieldArgs<float>& a) { return a.st->kick_f; }
__device__ __forceinline__ double kick_of(const FieldArgs<double>& a) { return a.st->kick; }

// Unevaluated sums h + l of FP32 pairs (|l| <= ulp(h)), about twice the working
// precision: FP64 runs at 1/64 of the FP32 rate here, and the some 17 FP64
// operations per particle that these pairs replace bound the field kernel at low
// degrees: N = 5e5, l_max = 1: 49.5 -> 33.9 us; N = 3e5, l_max = 8: 47.3 -> 44.2. The
// error of the inner charge is its last rounding, as with FP64: for N = 200 to 1.6e7 and
// r_out = 1.3 to 60 the rms error against extended precision is that of the FP64 form to
// a factor of 1.000002 (2.5e-8 of the rms charge; 0 to 2.5e-3 of the values differ, by a unit).
struct FF { float h, l; };
// a + b exactly (Knuth's TwoSum)
__device__ __forceinline__ FF ff_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fadd_rn(s, -a);
  return {s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb))};
}
// a b exactly
__device__ __forceinline__ FF ff_mul(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
// Ions of the uniform background inside the particle's radius: coef (r^3 - 1), with
// r = rf + corr by one Newton step from the FP32 root rf = r2 / r.
__device__ __forceinline__ FF uniform_ions_inside(float X, float Y, float Z, float ir, float coef_h, float coef_l) {
  const FF xx = ff_mul(X, X), yy = ff_mul(Y, Y), zz = ff_mul(Z, Z);
  const FF s1 = ff_sum(xx.h, yy.h), s2 = ff_sum(s1.h, zz.h);
  const float r2h = s2.h, r2l = s2.l + (s1.l + (xx.l + (yy.l + zz.l)));
  const float rf = __fmul_rn(r2h, ir);
  const float corr = (__fmaf_rn(-rf, rf, r2h) + r2l) * (0.5f * ir);
  const FF p = ff_mul(r2h, rf);  // r^3 = (r2h + r2l)(rf + corr)
  const FF d = ff_sum(p.h, -1.f);
  const float dl = d.l + (p.l + __fmaf_rn(r2h, corr, r2l * rf));
  const FF q = ff_mul(d.h, coef_h);
  return {q.h, q.l + __fmaf_rn(d.h, coef_l, dl * coef_h)};
}
// Ions of the radial profile (App. D) inside radius rd: linear between the
// nodes, constant outside [1, r_out].
template <class T> __device__ __forceinline__ double profile_ions_inside(const FieldArgs<T>& a, double rd) {
  const double t = fmin(fmax((rd - 1.0) * a.ion_inv_h, 0.0), double(a.ion_n - 1));
  const int k = min(int(t), a.ion_n - 2);
  const double q0 = __ldg(a.ion_q + k), q1 = __ldg(a.ion_q + k + 1);
  return a.ion_scale * fma(t - double(k), q1 - q0, q0);
}

// The rest of one particle's step, from the field E of the other particles' l >= 1
// terms: the l = 0 term, the own image, the push, the walls and collisions, the
// next radius key (or, in field mode, the field itself).
template <class T, int L>
__device__ __forceinline__ void field_finish(const FieldArgs<T>& a, int64_t j, bool valid, bool is_ion, T qneg, T X, T Y,
                                             T Z, T VX, T VY, T VZ, T r2, T ir2, T ir, T Ex, T Ey, T Ez, double qmob,
                                             double q_s, const uint32_t* id) {
  // l = 0: electrons inside (sorted index j), ions inside, surface charge;
  // then the self-image correction. The image moments of the far field sum
  // over all particles, the particle itself included, so without the self
  // image (self_image = 0) its own image field is taken off again; with
  // img_in_tile the own tile is left out of them, so with the self image
  // (self_image = 1) it is added. The count difference is small against its
  // terms: it is formed in twice the working precision from the exact r^2 of
  // the FP32 position (FP32 pairs), or in FP64.
  {
    T qin;  // inner charge in units of e: ions inside minus electrons inside (+ Q_S)
    if constexpr (sizeof(T) == 4) {
      if (!a.ion_q) {
        const FF qion = uniform_ions_inside(X, Y, Z, ir, a.ion_coef_h, a.ion_coef_l);
        FF mob;  // charge of the mobile particles inside: j electrons, or the species' scan
        if (a.species) {
          mob.h = float(qmob);
          mob.l = float(qmob - double(mob.h));
        } else {
          const uint32_t ju = uint32_t(j);  // j < N <= 2^31
          mob.h = -__uint2float_rn(ju);
          mob.l = a.n > (1 << 24) ? -float(int32_t(ju - __float2uint_rz(-mob.h))) : 0.f;
        }
        const FF d1 = ff_sum(qion.h, mob.h), d2 = ff_sum(d1.h, a.st->qs_h);
        qin = d2.h + (d2.l + (d1.l + (mob.l + (qion.l + a.st->qs_l))));
      } else {
        const double xd = double(X), yd = double(Y), zd = double(Z);
        const double r2d = xd * xd + yd * yd + zd * zd;  // exact for FP32 positions
        // FP32 root refined by one Newton step in FP64 (no FP64 sqrt or division)
        const float rf = r2 * ir;
        const double rd = double(rf) + (r2d - double(rf) * double(rf)) * double(0.5f * ir);
        qin = T(profile_ions_inside(a, rd) + (q_s + (a.species ? qmob : -double(int32_t(j)))));
      }
    } else {
      const double r2d = X * X + Y * Y + Z * Z, rd = sqrt(r2d);
      const double qion = a.ion_q ? profile_ions_inside(a, rd) : a.ion_coef * (r2d * rd - 1.0);
      qin = qion + (q_s + (a.species ? qmob : -double(int32_t(j))));
    }
    const T er = qin * (a.pf_t * ir2 * ir);  // multiplies x (gives r^ / r^2)
    Ex += er * X; Ey += er * Y; Ez += er * Z;
    const int self_sign = a.self_sign;
    if (self_sign != 0 && a.m0_only) {
      // own image with the m = 0 kernel: pf sum_l f_l r^{-(2l+3)} [(l+1) P_l^2 r^ - P_l P_l' (z^ - u r^)]
      const T u = Z * ir;
      T Pm = T(1), P = u, Dm = T(0), D = T(1), rp = ir2 * ir2 * ir;  // r^{-5} at l = 1
      T hr = T(0), ha = T(0);
#pragma unroll
      for (int l = 1; l <= L; ++l) {
        if (l > 1) {
          const T Pn = (T(2 * l - 1) * u * P - T(l - 1) * Pm) / T(l);
          const T Dn = Dm + T(2 * l - 1) * P;
          Pm = P; P = Pn; Dm = D; D = Dn;
          rp *= ir2;
        }
        hr += a.f[l] * T(l + 1) * P * P * rp;
        ha += a.f[l] * P * D * rp;
      }
      const T pfT = a.self_pf * qneg;
      // r^ = x / r, z^ - u r^ = (0, 0, 1) - u x / r
      Ex += pfT * (hr * X * ir + ha * u * X * ir);
      Ey += pfT * (hr * Y * ir + ha * u * Y * ir);
      Ez += pfT * (hr * Z * ir - ha * (T(1) - u * Z * ir));
    } else if (self_sign != 0) {
      // the particle's own image: pf sum_l f_l (l+1) r^{-(2l+3)} r^
      T h = T(0);
#pragma unroll
      for (int l = L; l >= 1; --l) h = h * ir2 + a.f[l] * T(l + 1);
      const T es = a.self_pf * qneg * h * ir2 * ir2 * ir2;  // r^{-(2l+3)} r^ = ir2^{l-1} ir2^3 x
      Ex += es * X; Ey += es * Y; Ez += es * Z;
    }
  }

  if (a.mode == 1) {
    if (valid) {
      a.Eout[j] = Ex;
      a.Eout[a.n + j] = Ey;
      a.Eout[2 * a.n + j] = Ez;
    }
    return;
  }
  if (!valid) return;

  const T kick = kick_of(a);
  // ---- leapfrog: v += kick (q/m) E (q/m = -1 for an electron); x += dt v
  if (is_ion) {
    const T kq = kick * a.qm_ion;
    VX += kq * Ex; VY += kq * Ey; VZ += kq * Ez;
  } else {
    VX -= kick * Ex; VY -= kick * Ey; VZ -= kick * Ez;
  }
  X += a.dt * VX; Y += a.dt * VY; Z += a.dt * VZ;

  // ---- walls (Sec. 4): mirror the radius back, keep the speed
  {
    double rr = 0.0;
    bool hit = false;
    {
      const T rt = X * X + Y * Y + Z * Z;
      const bool near_wall = rt < T(1.0 + 1e-5) || rt > a.near_hi;
      if (near_wall) {  // the exact test in FP64 only near a wall
        const double xd = double(X), yd = double(Y), zd = double(Z);
        rr = xd * xd + yd * yd + zd * zd;  // exact for FP32 positions
        hit = rr < 1.0 || rr > a.r_out2;
      }
    }
    if (hit && a.wall_rule == 2) {
      // absorbed (at the probe its charge joins Q_S) and replaced from the outer wall
      if (rr < 1.0) atomicAdd(a.nabs, 1);
      double xn[3], vn[3];
      inject_particle(*id, uint64_t(a.st->step), a.seed, double(a.r_out), double(a.dt), a.sigma_v, xn, vn);
      X = T(xn[0]); Y = T(xn[1]); Z = T(xn[2]);
      VX = T(vn[0]); VY = T(vn[1]); VZ = T(vn[2]);
    } else if (hit) {
      const double xd = double(X), yd = double(Y), zd = double(Z);
      const double rd = sqrt(rr);
      const bool inner = rr < 1.0;
      double rn = inner ? 2.0 - rd : 2.0 * double(a.r_out) - rd;
      rn = rn < 1.0 ? 1.0 : (rn > double(a.r_out) ? double(a.r_out) : rn);
      const double e0 = xd / rd, e1 = yd / rd, e2 = zd / rd;
      X = T(e0 * rn); Y = T(e1 * rn); Z = T(e2 * rn);
      if (a.wall_rule == 1) {
        const T vr = VX * T(e0) + VY * T(e1) + VZ * T(e2);
        VX -= T(2) * vr * T(e0); VY -= T(2) * vr * T(e1); VZ -= T(2) * vr * T(e2);
      } else {
        const T sgn = inner ? T(1) : T(-1);
        const T n0 = sgn * T(e0), n1 = sgn * T(e1), n2 = sgn * T(e2);
        const T speed = sqrt(VX * VX + VY * VY + VZ * VZ);
        const uint64_t stp = uint64_t(a.st->step);
        const uint4 o = philox4x32_10(
            make_uint4(uint32_t(stp), uint32_t(stp >> 32), *id, 0x494D5250u),
            make_uint2(uint32_t(a.seed), uint32_t(a.seed >> 32)));
        const T u1 = T(o.x >> 8) * T(1.0 / 16777216.0);
        const T u2 = T(o.y >> 8) * T(1.0 / 16777216.0);
        const T ca = T(1) - u1;
        const T sa = sqrt(T(1) - ca * ca);
        T sp, cp;
        if constexpr (sizeof(T) == 4) sincospif(T(2) * u2, &sp, &cp);
        else sincospi(T(2) * u2, &sp, &cp);
        const T sg = n2 >= T(0) ? T(1) : T(-1);
        const T aa = T(-1) / (sg + n2);
        const T bb = n0 * n1 * aa;
        const T t10 = T(1) + sg * n0 * n0 * aa, t11 = sg * bb, t12 = -sg * n0;
        const T t20 = bb, t21 = sg + n1 * n1 * aa, t22 = -n1;
        VX = speed * (ca * n0 + sa * (cp * t10 + sp * t20));
        VY = speed * (ca * n1 + sa * (cp * t11 + sp * t21));
        VZ = speed * (ca * n2 + sa * (cp * t12 + sp * t22));
      }
    }
    if (a.coll_thr != 0u && !is_ion) {
      // electron-neutral collision: isotropic elastic scattering with
      // probability 1 - exp(-nu dt) (Philox counter (step, step >> 32, id,
      // 0x434F4C4C), key = seed; top 24 bits below the threshold)
      const uint64_t stp = uint64_t(a.st->step);
      const uint4 o = philox4x32_10(make_uint4(uint32_t(stp), uint32_t(stp >> 32), *id, 0x434F4C4Cu),
                                    make_uint2(uint32_t(a.seed), uint32_t(a.seed >> 32)));
      if ((o.x >> 8) < a.coll_thr) {
        const T speed = sqrt(VX * VX + VY * VY + VZ * VZ);
        const T u1 = T(o.y >> 8) * T(1.0 / 16777216.0);
        const T u2 = T(o.z >> 8) * T(1.0 / 16777216.0);
        const T ct = T(1) - T(2) * u1;
        const T st = sqrt(T(1) - ct * ct);
        T sp, cp;
        if constexpr (sizeof(T) == 4) sincospif(T(2) * u2, &sp, &cp);
        else sincospi(T(2) * u2, &sp, &cp);
        VX = speed * st * cp;
        VY = speed * st * sp;
        VZ = speed * ct;
      }
    }
    const bool fin = isfinite(X) && isfinite(Y) && isfinite(Z) && isfinite(VX) && isfinite(VY) && isfinite(VZ);
    if (!fin) atomicOr(a.err, kErrNaN);
    a.key[j] = fin ? radius_key<T>(X, Y, Z, a.rk) : 0u;
    a.kidx[j] = uint32_t(j);
  }
  Part<T> rec;
  rec.x = X; rec.y = Y; rec.z = Z;
  rec.vx = VX; rec.vy = VY; rec.vz = VZ;
  rec.id = *id;
  a.out[j] = rec;
}

// One warp per tile. Phase 1 forms the tile's expansion coefficients, phase 2
// their gradients (ladder identities) in shared memory, phase 3 evaluates the
// far field of all other tiles, the near field of the pairs inside the tile,
// the l = 0 terms, and then pushes the particle.
// Body of the field kernel for warp `warp` of a CTA of `wpb` warps, tile
// `tile` of the instance whose arguments are `a`.
// IC: in FP32 the image pairs of the own tile that are summed together (img_in_tile); 0 leaves
// that code out.
template <class T, int L, int IC>
__device__ __forceinline__ void field_tile(const FieldArgs<T>& a, unsigned char* smem_raw, int warp, int wpb,
                                           int64_t tile) {
  using V4 = typename Vec4<T>::type;
  using V2 = typename Vec2<T>::type;
  constexpr int NC = 2 * ncomp(L);
  constexpr int NI = nI(L), NR = nR(L);
  constexpr int NE = NI + NR;
  const Tables<T>& tb = tab<T>();
  const unsigned lane = lane_id();
  const int64_t ntiles = (a.n + 31) >> 5;
  if (tile >= ntiles) return;  // warp-uniform; no block-wide barrier below
  const int64_t ts = tile_stride(ntiles);
  constexpr int CH = chunk_cap(L);
  V4* coefA = reinterpret_cast<V4*>(smem_raw) + size_t(warp) * CH;
  V2* coefB = reinterpret_cast<V2*>(reinterpret_cast<V4*>(smem_raw) + size_t(wpb) * CH) + size_t(warp) * CH;
  T* sc = reinterpret_cast<T*>(reinterpret_cast<V2*>(reinterpret_cast<V4*>(smem_raw) + size_t(wpb) * CH) +
                               size_t(wpb) * CH) + size_t(warp) * (NC + 2);
  const int64_t g = tile / kTilesPerGroup;
  const double q_s = a.q_s + a.st->qs_acc;  // with the charge absorbed at the probe so far
  const bool img_in_tile = IC > 0 && img_in_tile_for<T>(0) && a.img_in_tile;  // FP32 contexts only

  // the particle of this lane, loaded first so that its latency overlaps the
  // prologue
  const int64_t j = tile * 32 + lane;
  const bool valid = j < a.n;
  T X = valid ? a.x[j] : T(1), Y = valid ? a.y[j] : T(0), Z = valid ? a.z[j] : T(0);
  T VX = T(0), VY = T(0), VZ = T(0);
  if (a.mode == 0 && valid) { VX = a.vx[j]; VY = a.vy[j]; VZ = a.vz[j]; }
  // mobile ions: ids from n_e on are ions; qneg = -q (1 for an electron), 0 on an empty lane
  const bool is_ion = a.species && valid && a.id[j] >= a.n_e;
  const T qneg = valid ? (is_ion ? -a.q_ion : T(1)) : T(0);

  // ---- phase 1: cI (coefficients of Is, s = 0) and cR (of Rs(x/r_out), s = 1),
  // with the gradient's scale -pf (and 1/r_out for Rs) applied, and the zero slot.
  // The loop has a fixed trip count and is unrolled, so that all loads of the
  // scan carries are in flight at once.
  const T mpf = a.mpf, mpfr = a.mpfr;
  if (lane == 0) { sc[NC] = T(0); sc[NC + 1] = T(0); }
  {
    const V2* pt = reinterpret_cast<const V2*>(a.pfx + tile * NC);  // [tile][u]: (A, B) pairs
    const T* gb = a.gbase + g * NC;
    const T* at = a.agg + tile;   // [u][tile]
    const uint16_t* ctab = g_comp + comp_tab_off(L);
    constexpr int NIT = (NC / 2 + 31) / 32;
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      const int e = int(lane) + 32 * it;
      if (e < NC / 2) {
        const uint16_t cr = ctab[e];
        const int l = cr & 0xff;
        const T rl = a.rhol[l];  // r_out^l
        const V2 ab = pt[e];
        const T A = gb[2 * e] + ab.x;      // sum over inner tiles of q Rs(x_i / r_out)
        const T B = gb[2 * e + 1] + ab.y;  // sum over outer tiles of q Is(x_i)
        // sum of q Is(x_i) of the image term: over all particles, or over the
        // other tiles when the own tile's image pairs are summed directly
        const T W = img_in_tile ? a.tot[2 * e + 1] - at[(2 * e + 1) * ts] : a.tot[2 * e + 1];
        T cI = rl * A - a.f[l] * W;
        if ((cr >> 8) & 1) cI += drive_of(a, l);
        T cR = rl * B;
        if (a.m0_only && ((cr >> 9) & 1)) { cI = T(0); cR = T(0); }
        sc[2 * e] = cI * mpf;
        sc[2 * e + 1] = cR * mpfr;
      }
    }
  }
  __syncwarp();
  // ---- phase 3: the particle of this lane
  const T r2 = X * X + Y * Y + Z * Z;
  const T ir2 = T(1) / r2;
  const T ir = rsqrt_t(r2);
  T Ex = T(0), Ey = T(0), Ez = T(0);
  T Fx = T(0), Fy = T(0), Fz = T(0);  // second accumulator chain (Im parts)

  // ---- far field, in column chunks of at most kChunk gradient entries: the
  // entries of a chunk are formed in shared memory (phase 2) and evaluated at
  // once; the recurrence's diagonal term is carried from chunk to chunk in
  // registers.
  const EntryRec* etab = g_ent + ent_off(L);
  auto build = [&](int k0, int k1) {
    __syncwarp();
    constexpr int NB = (CH + 31) / 32;  // at most CH entries per build
#pragma unroll 1
    for (int it = 0; it < NB; ++it) {
      const int k = k0 + int(lane) + 32 * it;
      if (k < k1) {
        const EntryRec er = etab[k];
        const T c1r = sc[er.src[0]], c1i = sc[er.src[1]], c2r = sc[er.src[2]], c2i = sc[er.src[3]],
                c0r = sc[er.src[4]], c0i = sc[er.src[5]];
        const T s1r = T(er.s1r), s1i = T(er.s1i), s2 = T(er.s2), sz = T(er.sz);
        V4 ca;
        V2 cb;
        ca.x = s1r * c1r + s2 * c2r;  // d/dx, d/dy, d/dz (Re), d/dx (Im)
        ca.y = s2 * c2i - s1i * c1i;
        ca.z = sz * c0r;
        ca.w = s1i * c1i + s2 * c2i;
        cb.x = s1r * c1r - s2 * c2r;  // d/dy, d/dz (Im)
        cb.y = sz * c0i;
        coefA[k - k0] = ca;
        coefB[k - k0] = cb;
      }
    }
    __syncwarp();
  };

  if constexpr (!chunked(L)) build(0, NE);  // all entries of both parts at once
  // Two forms of the far-field loops, chosen per degree by measurement
  // (rolled_far): fully unrolled (compile-time coefficients and entry
  // addresses), or with the columns m >= 1 in a rolled loop (the recurrence
  // over l = m + j unrolled, with a uniform exit at the column end; the real
  // column m = 0 peeled), which keeps the code and the register count small.
  if constexpr (!rolled_far(L)) {
    // multipole part: sum over Is_l^m(x), 1 <= l <= L+1
    {
      const T Zir2 = Z * ir2;
      T dr = ir, di = T(0);
      constexpr int QI = chunked(L) ? nchunkI(L) : 1;
#pragma unroll
      for (int q = 0; q < QI; ++q) {
        const int m0 = chunked(L) ? chunkI(L, q) : 0, m1 = chunked(L) ? chunkI(L, q + 1) : L + 2;
        const int k0 = chunked(L) ? offI(L, m0) : 0;
        if constexpr (chunked(L)) build(k0, offI(L, m1));
#pragma unroll
        for (int m = m0; m < m1; ++m) {
          if (m > 0) {
            const T c = tb.dg[m];
            const T ex = c * X * ir2, ey = c * Y * ir2;
            const T nr = ex * dr - ey * di, ni = ex * di + ey * dr;
            dr = nr;
            di = ni;
          }
          // the column is (dr + i di) times the real p_l, which obeys the
          // same recurrence from p_m = 1: sum the contractions with p_l, then
          // multiply by the diagonal once per column
          T p1 = T(1), p0 = T(0);
          T Sx = T(0), Sy = T(0), Sz = T(0), Tx = T(0), Ty = T(0), Tz = T(0);
#pragma unroll
          for (int l = m; l <= L + 1; ++l) {
            if (l > m) {
              const T A = tb.an[l * kTabL + m] * Zir2;
              const T pn = A * p1 - ir2 * p0;
              p0 = p1; p1 = pn;
            }
            if (l >= 1) {
              const V4 ca = coefA[idxI(L, l, m) - k0];
              if (l == m) {
                Sx = ca.x; Sy = ca.y; Sz = ca.z;
              } else {
                Sx += ca.x * p1; Sy += ca.y * p1; Sz += ca.z * p1;
              }
              if (m > 0) {
                const V2 cb = coefB[idxI(L, l, m) - k0];
                if (l == m) {
                  Tx = ca.w; Ty = cb.x; Tz = cb.y;
                } else {
                  Tx += ca.w * p1; Ty += cb.x * p1; Tz += cb.y * p1;
                }
              }
            }
          }
          Ex += dr * Sx; Ey += dr * Sy; Ez += dr * Sz;
          if (m > 0) { Fx += di * Tx; Fy += di * Ty; Fz += di * Tz; }
        }
      }
    }
    // local part: sum over Rs_l^m(x / r_out), 0 <= l <= L-1
    {
      const T Xs = X * a.rho_inv, Ys = Y * a.rho_inv, Zs = Z * a.rho_inv;
      const T rs2 = r2 * a.rho_inv * a.rho_inv;
      T dr = T(1), di = T(0);
      constexpr int QR = chunked(L) ? nchunkR(L) : 1;
#pragma unroll
      for (int q = 0; q < QR; ++q) {
        const int m0 = chunked(L) ? chunkR(L, q) : 0, m1 = chunked(L) ? chunkR(L, q + 1) : L;
        const int k0 = chunked(L) ? NI + offR(L, m0) : 0;
        if constexpr (chunked(L)) build(k0, NI + offR(L, m1));
#pragma unroll
        for (int m = m0; m < m1; ++m) {
          if (m > 0) {
            const T c = tb.dg[m];
            const T ex = c * Xs, ey = c * Ys;
            const T nr = ex * dr - ey * di, ni = ex * di + ey * dr;
            dr = nr;
            di = ni;
          }
          T p1 = T(1), p0 = T(0);
          T Sx = T(0), Sy = T(0), Sz = T(0), Tx = T(0), Ty = T(0), Tz = T(0);
#pragma unroll
          for (int l = m; l <= L - 1; ++l) {
            if (l > m) {
              const T A = tb.an[l * kTabL + m] * Zs;
              const T pn = A * p1 - rs2 * p0;
              p0 = p1; p1 = pn;
            }
            const V4 ca = coefA[NI + idxR(L, l, m) - k0];
            if (l == m) {
              Sx = ca.x; Sy = ca.y; Sz = ca.z;
            } else {
              Sx += ca.x * p1; Sy += ca.y * p1; Sz += ca.z * p1;
            }
            if (m > 0) {
              const V2 cb = coefB[NI + idxR(L, l, m) - k0];
              if (l == m) {
                Tx = ca.w; Ty = cb.x; Tz = cb.y;
              } else {
                Tx += ca.w * p1; Ty += cb.x * p1; Tz += cb.y * p1;
              }
            }
          }
          Ex += dr * Sx; Ey += dr * Sy; Ez += dr * Sz;
          if (m > 0) { Fx += di * Tx; Fy += di * Ty; Fz += di * Tz; }
        }
      }
    }

  } else {
    // multipole part: sum over Is_l^m(x), 1 <= l <= L+1
    {
      const T Zir2 = Z * ir2;
      T dr = ir, di = T(0);
      constexpr int QI = chunked(L) ? nchunkI(L) : 1;
#pragma unroll
      for (int q = 0; q < QI; ++q) {
        const int m0 = chunked(L) ? chunkI(L, q) : 0, m1 = chunked(L) ? chunkI(L, q + 1) : L + 2;
        const int k0 = chunked(L) ? offI(L, m0) : 0;
        if constexpr (chunked(L)) build(k0, offI(L, m1));
        if (m0 == 0) {
          T c1 = dr, c0 = T(0);
#pragma unroll
          for (int l = 1; l <= L + 1; ++l) {
            const T A = tb.an[l * kTabL] * Zir2, B = ir2;
            const T n1 = A * c1 - B * c0;
            c0 = c1; c1 = n1;
            const V4 ca = coefA[idxI(L, l, 0) - k0];
            Ex += ca.x * c1; Ey += ca.y * c1; Ez += ca.z * c1;
          }
        }
  #pragma unroll 1
        for (int m = m0 > 1 ? m0 : 1; m < m1; ++m) {
          const T c = tb.dg[m];
          {
            const T ex = c * X * ir2, ey = c * Y * ir2;
            const T nr = ex * dr - ey * di, ni = ex * di + ey * dr;
            dr = nr;
            di = ni;
          }
          const int eb = offI(L, m) - k0 - (m > 1 ? m : 1);  // entry of degree l: eb + l
          T cA[L + 1];  // the column's recurrence coefficients, loaded before its steps
#pragma unroll
          for (int j = 1; j <= L; ++j) cA[j] = m + j <= L + 1 ? tb.an[(m + j) * kTabL + m] : T(0);
          T p1 = T(1), p0 = T(0);  // the column is (dr + i di) p_l
          T Sx, Sy, Sz, Tx, Ty, Tz;
          {
            const V4 ca = coefA[eb + m];
            const V2 cb = coefB[eb + m];
            Sx = ca.x; Sy = ca.y; Sz = ca.z;
            Tx = ca.w; Ty = cb.x; Tz = cb.y;
          }
#pragma unroll
          for (int j = 1; j <= L; ++j) {
            const int l = m + j;
            if (l > L + 1) break;
            const T A = cA[j] * Zir2;
            const T pn = A * p1 - ir2 * p0;
            p0 = p1; p1 = pn;
            const V4 ca = coefA[eb + l];
            const V2 cb = coefB[eb + l];
            Sx += ca.x * p1; Sy += ca.y * p1; Sz += ca.z * p1;
            Tx += ca.w * p1; Ty += cb.x * p1; Tz += cb.y * p1;
          }
          Ex += dr * Sx; Ey += dr * Sy; Ez += dr * Sz;
          Fx += di * Tx; Fy += di * Ty; Fz += di * Tz;
        }
      }
    }
    // local part: sum over Rs_l^m(x / r_out), 0 <= l <= L-1
    {
      const T Xs = X * a.rho_inv, Ys = Y * a.rho_inv, Zs = Z * a.rho_inv;
      const T rs2 = r2 * a.rho_inv * a.rho_inv;
      T dr = T(1), di = T(0);
      constexpr int QR = chunked(L) ? nchunkR(L) : 1;
#pragma unroll
      for (int q = 0; q < QR; ++q) {
        const int m0 = chunked(L) ? chunkR(L, q) : 0, m1 = chunked(L) ? chunkR(L, q + 1) : L;
        const int k0 = chunked(L) ? NI + offR(L, m0) : 0;
        if constexpr (chunked(L)) build(k0, NI + offR(L, m1));
        if (m0 == 0) {
          T c1 = dr, c0 = T(0);
#pragma unroll
          for (int l = 0; l <= L - 1; ++l) {
            if (l > 0) {
              const T A = tb.an[l * kTabL] * Zs, B = rs2;
              const T n1 = A * c1 - B * c0;
              c0 = c1; c1 = n1;
            }
            const V4 ca = coefA[NI + idxR(L, l, 0) - k0];
            Ex += ca.x * c1; Ey += ca.y * c1; Ez += ca.z * c1;
          }
        }
  #pragma unroll 1
        for (int m = m0 > 1 ? m0 : 1; m < m1; ++m) {
          const T c = tb.dg[m];
          {
            const T ex = c * Xs, ey = c * Ys;
            const T nr = ex * dr - ey * di, ni = ex * di + ey * dr;
            dr = nr;
            di = ni;
          }
          const int eb = NI + offR(L, m) - k0 - m;  // entry of degree l: eb + l
          T cA[L];  // the column's recurrence coefficients, loaded before its steps
#pragma unroll
          for (int j = 1; j <= L - 1; ++j) cA[j] = m + j <= L - 1 ? tb.an[(m + j) * kTabL + m] : T(0);
          T p1 = T(1), p0 = T(0);
          T Sx, Sy, Sz, Tx, Ty, Tz;
          {
            const V4 ca = coefA[eb + m];
            const V2 cb = coefB[eb + m];
            Sx = ca.x; Sy = ca.y; Sz = ca.z;
            Tx = ca.w; Ty = cb.x; Tz = cb.y;
          }
#pragma unroll
          for (int j = 1; j <= L - 1; ++j) {
            const int l = m + j;
            if (l > L - 1) break;
            const T A = cA[j] * Zs;
            const T pn = A * p1 - rs2 * p0;
            p0 = p1; p1 = pn;
            const V4 ca = coefA[eb + l];
            const V2 cb = coefB[eb + l];
            Sx += ca.x * p1; Sy += ca.y * p1; Sz += ca.z * p1;
            Tx += ca.w * p1; Ty += cb.x * p1; Tz += cb.y * p1;
          }
          Ex += dr * Sx; Ey += dr * Sy; Ez += dr * Sz;
          Fx += di * Tx; Fy += di * Ty; Fz += di * Tz;
        }
      }
    }

  }
  Ex += Fx; Ey += Fy; Ez += Fz;

  // near field: the direct pair terms r_<^l / r_>^{l+1} P_l (l >= 1) of the
  // particles of this tile (their image terms are separable and are part of
  // the far field). Lower lane = smaller sorted radius = inner.
  {
    const T rk = r2 * ir;
    const T ex = X * ir, ey = Y * ir, ez = Z * ir;
    T Nx = T(0), Ny = T(0), Nz = T(0);  // sum of grad phi (phi = sum_l r_<^l/r_>^{l+1} P_l), weighted by -q
    // -q of this particle (1 for an electron), 0 for the empty lanes of a
    // ragged tile: a partner's contribution to my field is weighted by its
    // -q (pm), mine to the partner's by vmask
    const T vmask = qneg;
#pragma unroll 1
    for (int s = 1; s <= 16 && !a.m0_only; ++s) {
      const int src = (lane + s) & 31;
      const T pex = __shfl_sync(0xffffffffu, ex, src);
      const T pey = __shfl_sync(0xffffffffu, ey, src);
      const T pez = __shfl_sync(0xffffffffu, ez, src);
      const T prk = __shfl_sync(0xffffffffu, rk, src);
      const T pir = __shfl_sync(0xffffffffu, ir, src);
      const T pm = __shfl_sync(0xffffffffu, vmask, src);
      const bool me_inner = int(lane) < src;
      const T sr = me_inner ? rk * pir : prk * ir;  // r_inner / r_outer
      const T uu = ex * pex + ey * pey + ez * pez;
      // Q_l = s^l P_l(u) and E_l = s^(l-1) P'_l(u), scaled (leg_c, leg_eps) so
      // that each step is one product with a per-degree constant less:
      // S0 = sum Q_l, S1 = sum l Q_l, S2 = sum s E_l = sum s^l P'_l(u).
      const T x1 = sr * uu, y2 = sr * sr;
      T qm = T(1), q = x1, em = T(0), e = T(1);
      T S0 = x1, S1 = x1, S2 = T(1);
#pragma unroll
      for (int l = 1; l < L; ++l) {
        const T qn = fma_t(x1, q, -(T(leg_g(l)) * y2) * qm);
        const T en = l == 1 ? q : fma_t(T(leg_r(l)) * y2, em, q);
        qm = q; q = qn; em = e; e = en;
        S0 = fma_t(T(leg_c(l + 1)), q, S0);
        S1 = fma_t(T((l + 1) * leg_c(l + 1)), q, S1);
        S2 = fma_t(T(leg_eps(l + 1)), e, S2);
      }
      S2 *= sr;
      // grad of phi = sum_l r_i^l/r_o^{l+1} P_l(u): at the inner end
      // (S1 r^_i + S2 (r^_o - u r^_i)) / (r_i r_o), at the outer end
      // (-(S0 + S1) r^_o + S2 (r^_i - u r^_o)) / r_o^2; radial (r) and angular
      // (a) factors of my end and of the partner's, with the validity mask
      const T gab = ir * pir;                          // 1 / (r_i r_o)
      const T go2 = me_inner ? pir * pir : ir * ir;    // 1 / r_o^2
      const T in_r = S1 * gab, in_a = S2 * gab;
      const T out_r = -(S0 + S1) * go2, out_a = S2 * go2;
      const T mr = (me_inner ? in_r : out_r) * pm, ma = (me_inner ? in_a : out_a) * pm;
      Nx += mr * ex + ma * (pex - uu * ex);
      Ny += mr * ey + ma * (pey - uu * ey);
      Nz += mr * ez + ma * (pez - uu * ez);
      if (s < 16) {
        const T pr = (me_inner ? out_r : in_r) * vmask, pa = (me_inner ? out_a : in_a) * vmask;
        const T tx = pr * pex + pa * (ex - uu * pex), ty = pr * pey + pa * (ey - uu * pey),
                tz = pr * pez + pa * (ez - uu * pez);
        const int dst = (lane - s) & 31;
        Nx += __shfl_sync(0xffffffffu, tx, dst);
        Ny += __shfl_sync(0xffffffffu, ty, dst);
        Nz += __shfl_sync(0xffffffffu, tz, dst);
      }
    }
#pragma unroll 1
    for (int s = 1; s <= 16 && a.m0_only; ++s) {
      // m = 0 truncation: sum_l r_i^l / r_o^{l+1} P_l(cos t_i) P_l(cos t_o)
      const int src = (lane + s) & 31;
      const T pex = __shfl_sync(0xffffffffu, ex, src);
      const T pey = __shfl_sync(0xffffffffu, ey, src);
      const T pez = __shfl_sync(0xffffffffu, ez, src);
      const T prk = __shfl_sync(0xffffffffu, rk, src);
      const T pir = __shfl_sync(0xffffffffu, ir, src);
      const T pm = __shfl_sync(0xffffffffu, vmask, src);
      const bool me_inner = int(lane) < src;
      const T ri = me_inner ? rk : prk;
      const T iri = me_inner ? ir : pir, iro = me_inner ? pir : ir;
      const T xix = me_inner ? ex : pex, xiy = me_inner ? ey : pey, xiz = me_inner ? ez : pez;
      const T xox = me_inner ? pex : ex, xoy = me_inner ? pey : ey, xoz = me_inner ? pez : ez;
      const T sr = ri * iro;
      const T ui = xiz, uo = xoz;  // cos of the polar angles
      T Pim = T(1), Pi = ui, Dim = T(0), Di = T(1);
      T Pom = T(1), Po = uo, Dom = T(0), Do = T(1);
      T sp = sr;  // s^l at l = 1
      T A1 = T(0), A3 = T(0), C1 = T(0), C2 = T(0);
#pragma unroll
      for (int l = 1; l <= L; ++l) {
        if (l > 1) {
          const T cl = T(2 * l - 1) / T(l), dl = T(l - 1) / T(l);
          const T Pin = cl * ui * Pi - dl * Pim, Pon = cl * uo * Po - dl * Pom;
          const T Din = Dim + T(2 * l - 1) * Pi, Don = Dom + T(2 * l - 1) * Po;
          Pim = Pi; Pi = Pin; Dim = Di; Di = Din;
          Pom = Po; Po = Pon; Dom = Do; Do = Don;
          sp *= sr;
        }
        const T pp = Pi * Po;
        A1 += T(l + 1) * sp * pp;
        A3 += T(l) * sp * pp;
        const T wgt = sp * iro;
        C1 += wgt * Pi * Do;
        C2 += wgt * Di * Po;
      }
      // grad at the outer point and at the inner point
      const T go = -A1 * iro * iro, gi = A3 * iro * iri;
      const T ogx = go * xox - C1 * iro * uo * xox, ogy = go * xoy - C1 * iro * uo * xoy,
              ogz = go * xoz + C1 * iro * (T(1) - uo * xoz);
      const T igx = gi * xix - C2 * iri * ui * xix, igy = gi * xiy - C2 * iri * ui * xiy,
              igz = gi * xiz + C2 * iri * (T(1) - ui * xiz);
      Nx += pm * (me_inner ? igx : ogx); Ny += pm * (me_inner ? igy : ogy); Nz += pm * (me_inner ? igz : ogz);
      if (s < 16) {
        const T tx = vmask * (me_inner ? ogx : igx), ty = vmask * (me_inner ? ogy : igy),
                tz = vmask * (me_inner ? ogz : igz);
        const int dst = (lane - s) & 31;
        Nx += __shfl_sync(0xffffffffu, tx, dst);
        Ny += __shfl_sync(0xffffffffu, ty, dst);
        Nz += __shfl_sync(0xffffffffu, tz, dst);
      }
    }
    if (img_in_tile) {
      // image terms of the other particles of the tile: grad at x_k of
      // -sum_l f_l P_l(u) / (r_k r_i)^{l+1}, u = x^_k . x^_i (m0_only:
      // P_l(cos t_k) P_l(cos t_i) in place of P_l(u)); d is the direction
      // along which u varies (x^_i, or z^ for m0_only)
      constexpr int C = IC > 0 ? IC : 1;
      T Gx = T(0), Gy = T(0), Gz = T(0);
#pragma unroll 1
      for (int s0 = 1; s0 < 32; s0 += C) {
        T pm[C], uu[C], dx[C], dy[C], dz[C], pz[C], tau[C], tp[C], Pm[C], P[C], Dm[C], D[C], Qm[C], Q[C], hr[C], ha[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const int src = (lane + s0 + c) & 31;
          const T pex = __shfl_sync(0xffffffffu, ex, src), pey = __shfl_sync(0xffffffffu, ey, src);
          pz[c] = __shfl_sync(0xffffffffu, ez, src);
          tau[c] = ir * __shfl_sync(0xffffffffu, ir, src);
          const T w = __shfl_sync(0xffffffffu, vmask, src);
          pm[c] = s0 + c < 32 ? w : T(0);
          uu[c] = a.m0_only ? ez : fma_t(ez, pz[c], fma_t(ey, pey, ex * pex));
          dx[c] = a.m0_only ? T(0) : pex; dy[c] = a.m0_only ? T(0) : pey; dz[c] = a.m0_only ? T(1) : pz[c];
          Pm[c] = T(1); P[c] = uu[c]; Dm[c] = T(0); D[c] = T(1);  // P_l(uu), P'_l(uu)
          Qm[c] = T(1); Q[c] = a.m0_only ? pz[c] : T(1);          // P_l(cos t_i) (m0_only), else 1
          tp[c] = tau[c] * tau[c];                                // tau^{l+1}
          hr[c] = ha[c] = T(0);
        }
#pragma unroll 1
        for (int l = 1; l <= L; ++l) {
          const T fl = a.f[l], cl = T(2 * l - 1) / T(l), dl = T(l - 1) / T(l);
          if (l > 1) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
              const T Pn = fma_t(cl * uu[c], P[c], -(dl * Pm[c])), Dn = fma_t(T(2 * l - 1), P[c], Dm[c]);
              Pm[c] = P[c]; P[c] = Pn; Dm[c] = D[c]; D[c] = Dn;
              if (a.m0_only) {
                const T Qn = fma_t(cl * pz[c], Q[c], -(dl * Qm[c]));
                Qm[c] = Q[c]; Q[c] = Qn;
              }
              tp[c] *= tau[c];
            }
          }
#pragma unroll
          for (int c = 0; c < C; ++c) {
            const T wgt = fl * tp[c] * Q[c];
            hr[c] = fma_t(T(l + 1) * wgt, P[c], hr[c]);
            ha[c] = fma_t(wgt, D[c], ha[c]);
          }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
          Gx = fma_t(pm[c], fma_t(hr[c], ex, -(ha[c] * fma_t(-uu[c], ex, dx[c]))), Gx);
          Gy = fma_t(pm[c], fma_t(hr[c], ey, -(ha[c] * fma_t(-uu[c], ey, dy[c]))), Gy);
          Gz = fma_t(pm[c], fma_t(hr[c], ez, -(ha[c] * fma_t(-uu[c], ez, dz[c]))), Gz);
        }
      }
      Nx += ir * Gx; Ny += ir * Gy; Nz += ir * Gz;
    }
    // E = -pf sum_i q_i grad phi (N holds the sum weighted by -q_i)
    const T pfT = a.pf_t;
    Ex += pfT * Nx; Ey += pfT * Ny; Ez += pfT * Nz;
  }

  double qmob = 0.0;  // with mobile ions: the charge of the particles inside (sorted before this one)
  if (a.species) {
    double qc = valid ? -double(qneg) : 0.0, incl = qc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, d);
      if (int(lane) >= d) incl += t;
    }
    qmob = a.qgbase[g] + a.qpfx[tile] + (incl - qc);
  }
  field_finish<T, L>(a, j, valid, is_ion, qneg, X, Y, Z, VX, VY, VZ, r2, ir2, ir, Ex, Ey, Ez, qmob, q_s, a.id + j);
}

// ----------------------------------------------------------------------------
// Field kernel of large FP32 instances of degree 12 and up (field_pair_rule): one
// warp per pair of tiles, half a warp per tile, two particles per lane (a: positions
// 0..15 of the tile, b: 16..31). field_tile is bound by issue slots (77 % busy, FMA
// pipe 52 %) and shared-memory wavefronts (58 %). Here the far field advances the
// multipole and the local harmonic of an (l, m) in one instruction (their recurrence
// shares its coefficients, their gradient factors lie side by side), one load serves
// two particles, and the near field takes two pairs per instruction: 5670 instructions
// per tile against 8370, FMA pipe 61 %, issue 60 % (ncu, N = 1e6, l_max = 16). The near
// field runs first, while the scan carries, velocities and ids are copied to shared
// memory. Field ms, field_tile -> this: l_max = 16, N = 2e6: 0.535 -> 0.470; l_max = 24,
// N = 4e6: 2.376 -> 1.843; l_max = 12, N = 7e5: 0.153 -> 0.128; l_max = 8, N = 2e6: 0.227 ->
// 0.224, l_max = 4: 0.145 -> 0.150 (not instantiated below 12).
// ----------------------------------------------------------------------------
// Two FP32 values advanced by one instruction.
__device__ __forceinline__ float2 f2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return f2(-a.x, -a.y); }
__device__ __forceinline__ float2 sel2(bool p, float2 a, float2 b) { return f2(p ? a.x : b.x, p ? a.y : b.y); }

// Constants of pair_sums, twice each: leg_c(l), l leg_c(l), -leg_g(l + 1).
struct __align__(16) LegRec { float2 c, lc, g, pad; };
struct LegTab { LegRec r[kTabL]; };
constexpr LegTab leg_tab() {
  LegTab t{};
  for (int l = 0; l < kTabL; ++l) {
    const float c = float(leg_c(l)), lc = float(l * leg_c(l)), g = float(-leg_g(l + 1));
    if (l == 0) { t.r[l] = LegRec{float2{0.f, 0.f}, float2{0.f, 0.f}, float2{g, g}, float2{0.f, 0.f}}; continue; }
    t.r[l] = LegRec{float2{c, c}, float2{lc, lc}, float2{g, g}, float2{0.f, 0.f}};
  }
  return t;
}
static __constant__ LegTab c_leg = leg_tab();

// The pair sums at (x1, y2) = (s u, s^2), s = r_inner / r_outer, u the cosine
// between the two: S0 = sum_{l=1..L} s^l P_l(u), S1 = sum l s^l P_l(u),
// S2 = sum s^(l-1) P'_l(u), by Clenshaw's backward recurrence for the monic
// polynomials q_l = s^l P_l / c_l (leg_g, leg_c) and its derivative in x1:
// 7 operations per degree (the forward recurrences of q_l and P'_l and three
// sums take 8), the same rounding error. Two sets of two pairs at once.
template <int L>
__device__ __forceinline__ void pair_sums(const float2 (&x1)[2], const float2 (&y2)[2], float2 (&S0)[2],
                                          float2 (&S1)[2], float2 (&S2)[2]) {
  float2 b2[2], d2[2], e2[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    S0[k] = f2(float(leg_c(L)));
    S1[k] = f2(float(L * leg_c(L)));
    S2[k] = b2[k] = d2[k] = e2[k] = f2(0.f);
  }
  constexpr int kUnr = L == 12 ? 12 : 8;  // l_max = 12: 0.128 ms with 12, 0.133 with 8 (N = 7e5)
#pragma unroll kUnr
  for (int l = L - 1; l >= 0; --l) {
    const LegRec r = c_leg.r[l];  // c = lc = 0 at l = 0
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float2 G = mul2(r.g, y2[k]);
      const float2 nb = fma2(x1[k], S0[k], fma2(G, b2[k], r.c)), nd = fma2(x1[k], S1[k], fma2(G, d2[k], r.lc)),
                   ne = fma2(x1[k], S2[k], fma2(G, e2[k], S0[k]));
      b2[k] = S0[k]; S0[k] = nb;
      d2[k] = S1[k]; S1[k] = nd;
      e2[k] = S2[k]; S2[k] = ne;
    }
  }
}

// Records of a tile built at once, in chunks of whole columns of at most this many:
// enough warps stay resident (l_max = 16 at N = 2e6, field ms: 96 gives 0.470 with 14
// warps per SM, 128 0.515, 80 0.479 with one chunk more).
constexpr int kPairCap = 96;
__host__ __device__ constexpr int pair_cap(int L) { return kPairCap < nP(L) ? kPairCap : nP(L); }
__host__ __device__ constexpr int pair_chunk(int L, int q) {  // first column of chunk q
  int m = 0;
  for (int c = 0; c < q && m <= L + 1; ++c) {
    int acc = 0;
    while (m <= L + 1 && acc + L + 2 - m <= pair_cap(L)) acc += L + 2 - m++;
  }
  return m;
}
__host__ __device__ constexpr int pair_nchunk(int L) {
  int q = 0;
  while (pair_chunk(L, q) <= L + 1) ++q;
  return q;
}
__host__ __device__ constexpr int pair_most(int L) {  // records of the largest chunk
  int most = 0;
  for (int q = 0; q < pair_nchunk(L); ++q) {
    const int n = offP(L, pair_chunk(L, q + 1)) - offP(L, pair_chunk(L, q));
    most = n > most ? n : most;
  }
  return most;
}
// float4s of a tile's records (three each), so that the two tiles start half a
// bank row apart (the two halves of a warp read different addresses at once).
__host__ __device__ constexpr int pair_stride(int L) { return (3 * pair_most(L) + 3) / 8 * 8 + 4; }
// The near field's particle data of the two tiles (over the entries, which are
// done with by then): 16 records of 12 + 12 + 8 floats per tile.
constexpr int kPairNear = 2 * 16 * 32 * 4;
// Words of one tile's complex coefficients and their zero slot (first its row of
// scan carries), and of the staged velocities, ids and positions of the two tiles.
__host__ __device__ constexpr int pair_row(int L) { return (4 * pair_run(L) + 2 + 3) / 4 * 4; }
constexpr int kPairVel = 7 * 64;
__host__ __device__ constexpr size_t pair_smem_per_warp(int L) {
  const size_t ent = size_t(2) * 16 * pair_stride(L);
  return (ent > size_t(kPairNear) ? ent : size_t(kPairNear)) + size_t(4) * (2 * pair_row(L) + kPairVel);
}
// Asynchronous copies of 4, 8 or 16 bytes from global to shared memory.
template <int B> __device__ __forceinline__ void copy_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src),
               "n"(B)
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int L>
__device__ __forceinline__ void field_pair(const FieldArgs<float>& a, unsigned char* smem_raw, int warp, int64_t pr) {
  constexpr int NC = 2 * ncomp(L), SR = pair_stride(L);
  const Tables<float>& tb = tab<float>();
  const int lane = int(lane_id()), h = lane >> 4, i = lane & 15;
  const int64_t ntiles = (a.n + 31) >> 5;
  if (2 * pr >= ntiles) return;  // warp-uniform; no block-wide barrier below
  unsigned char* const base = smem_raw + size_t(warp) * pair_smem_per_warp(L);
  float4* const rec0 = reinterpret_cast<float4*>(base);
  constexpr int SCW = pair_row(L);
  float* const sc0 = reinterpret_cast<float*>(base + pair_smem_per_warp(L)) - (2 * SCW + kPairVel);
  float* const vel = sc0 + 2 * SCW;  // [vx, vy, vz, id, x, y, z][64]
  const int64_t g = 2 * pr / kTilesPerGroup;  // both tiles lie in one group
  const int64_t tile = 2 * pr + h;
  const double q_s = a.q_s + a.st->qs_acc;

  int64_t j[2];
  bool valid[2];
  float X[2], Y[2], Z[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    j[p] = tile * 32 + 16 * p + i;
    valid[p] = j[p] < a.n;
    X[p] = valid[p] ? a.x[j[p]] : a.r_out;  // empty places count as outermost (weight 0)
    Y[p] = valid[p] ? a.y[j[p]] : 0.f;
    Z[p] = valid[p] ? a.z[j[p]] : 0.f;
  }

  // the scan carries of both tiles, the velocities and ids: copied to shared memory
  // while the near field computes
  {
    constexpr int B = NC % 4 == 0 ? 16 : 8, PER = NC * 4 / B;  // pieces of a row
    const char* src = reinterpret_cast<const char*>(a.pfx + 2 * pr * NC);
    char* const dst = reinterpret_cast<char*>(sc0);
#pragma unroll
    for (int k = 0; k < 2 * PER; k += 32) {
      const int c = k + lane;
      if (c < 2 * PER) copy_async<B>(dst + (c >= PER ? c - PER : c) * B + (c >= PER ? SCW * 4 : 0), src + c * B);
    }
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int o = 32 * h + 16 * p + i;
      vel[256 + o] = X[p]; vel[320 + o] = Y[p]; vel[384 + o] = Z[p];
      if (valid[p]) {
        copy_async<4>(vel + o, a.vx + j[p]);
        copy_async<4>(vel + 64 + o, a.vy + j[p]);
        copy_async<4>(vel + 128 + o, a.vz + j[p]);
        copy_async<4>(vel + 192 + o, a.id + j[p]);
      }
    }
  }

  float r2[2], ir[2];
  float2 E[2][3];  // the field: near field and multipole part, local part
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    r2[p] = X[p] * X[p] + Y[p] * Y[p] + Z[p] * Z[p];
    ir[p] = rsqrtf(r2[p]);
  }

  // near field: the pairs inside each tile. Lane i of a tile holds a_i and b_i
  // (a inner, b outer); in round t it takes (a_i, b_{i+t}) with (a_i, b_{i+t+8}), and
  // (a_i, a_{i+t+1}) with (b_i, b_{i+t+1}), two pairs per instruction. The other
  // end's factors go back to their lane, which applies them to the sender's
  // direction.
  float qneg[2];
  bool is_ion[2];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    is_ion[p] = a.species && valid[p] && a.id[j[p]] >= a.n_e;
    qneg[p] = valid[p] ? (is_ion[p] ? -a.q_ion : 1.f) : 0.f;
  }
  {
    float* const nb = reinterpret_cast<float*>(base) + h * (16 * 32);
    float4* const PB = reinterpret_cast<float4*>(nb);            // [16][3]: (b_j, b_{j+8}) x, y, z, r, 1/r, w
    float4* const PA = reinterpret_cast<float4*>(nb + 16 * 12);  // [16][3]: (a_j, b_j)
    float4* const PC = reinterpret_cast<float4*>(nb + 16 * 24);  // [16][2]: (a_j, a_{j+8}) x, y, z
    const float2 ux = f2(X[0] * ir[0], X[1] * ir[1]), uy = f2(Y[0] * ir[0], Y[1] * ir[1]),
                 uz = f2(Z[0] * ir[0], Z[1] * ir[1]), rk = f2(r2[0] * ir[0], r2[1] * ir[1]);
    {
      PA[3 * i] = make_float4(ux.x, ux.y, uy.x, uy.y);
      PA[3 * i + 1] = make_float4(uz.x, uz.y, rk.x, rk.y);
      PA[3 * i + 2] = make_float4(ir[0], ir[1], qneg[0], qneg[1]);
      const int i8 = (i + 8) & 15;
      float* const pb = nb;
      float* const pc = nb + 16 * 24;
      pb[12 * i + 0] = ux.y; pb[12 * i + 2] = uy.y; pb[12 * i + 4] = uz.y;
      pb[12 * i + 6] = rk.y; pb[12 * i + 8] = ir[1]; pb[12 * i + 10] = qneg[1];
      pb[12 * i8 + 1] = ux.y; pb[12 * i8 + 3] = uy.y; pb[12 * i8 + 5] = uz.y;
      pb[12 * i8 + 7] = rk.y; pb[12 * i8 + 9] = ir[1]; pb[12 * i8 + 11] = qneg[1];
      pc[8 * i + 0] = ux.x; pc[8 * i + 2] = uy.x; pc[8 * i + 4] = uz.x;
      pc[8 * i8 + 1] = ux.x; pc[8 * i8 + 3] = uy.x; pc[8 * i8 + 5] = uz.x;
    }
    __syncwarp();
    const float2 irab = f2(ir[0], ir[1]), w = f2(qneg[0], qneg[1]);
    // sums of -q grad phi: along the own direction (al) and the rest; of a (halves
    // of the rounds), of b (halves) and of (a, b)
    float2 aN[4] = {f2(0.f), f2(0.f), f2(0.f), f2(0.f)}, bN[4] = {f2(0.f), f2(0.f), f2(0.f), f2(0.f)},
           cN[4] = {f2(0.f), f2(0.f), f2(0.f), f2(0.f)};
    constexpr unsigned M = 0xffffffffu;
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
      // set 0: (a_i, b_{i+t}), (a_i, b_{i+t+8}), a the inner end; set 1:
      // (a_i, a_{i+t+1}), (b_i, b_{i+t+1})
      const int js0 = (i + t) & 15, js1 = (i + t + 1) & 15;
      const bool me_inner = i < js1;
      const float4 q0 = PB[3 * js0], q1 = PB[3 * js0 + 1], q2 = PB[3 * js0 + 2];
      const float4 o0 = PA[3 * js1], o1 = PA[3 * js1 + 1], o2 = PA[3 * js1 + 2];
      const float2 px[2] = {f2(q0.x, q0.y), f2(o0.x, o0.y)}, py[2] = {f2(q0.z, q0.w), f2(o0.z, o0.w)},
                   pz[2] = {f2(q1.x, q1.y), f2(o1.x, o1.y)}, pir[2] = {f2(q2.x, q2.y), f2(o2.x, o2.y)},
                   pw[2] = {f2(q2.z, q2.w), f2(o2.z, o2.w)};
      const float2 u[2] = {fma2(f2(ux.x), px[0], fma2(f2(uy.x), py[0], mul2(f2(uz.x), pz[0]))),
                           fma2(ux, px[1], fma2(uy, py[1], mul2(uz, pz[1])))};
      const float2 iro1 = sel2(me_inner, pir[1], irab);
      const float2 sr[2] = {mul2(f2(rk.x), pir[0]), mul2(sel2(me_inner, rk, f2(o1.z, o1.w)), iro1)};
      float2 S0[2], S1[2], S2[2];
      {
        const float2 x1[2] = {mul2(sr[0], u[0]), mul2(sr[1], u[1])}, y2[2] = {mul2(sr[0], sr[0]), mul2(sr[1], sr[1])};
        pair_sums<L>(x1, y2, S0, S1, S2);
      }
      // gradient of phi = sum_l r_i^l / r_o^{l+1} P_l(u): at the inner end
      // (S1 - u S') gab e_i + S' gab e_o, at the outer end -(S0 + S1 + u S') go2 e_o +
      // S' go2 e_i, with S' = s S2, gab = 1 / (r_i r_o), go2 = 1 / r_o^2
      float2 cin[2], cout[2], Sp[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        Sp[k] = mul2(S2[k], sr[k]);
        cin[k] = fma2(neg2(u[k]), Sp[k], S1[k]);
        cout[k] = neg2(fma2(u[k], Sp[k], add2(S0[k], S1[k])));
      }
      {
        const float2 gi = mul2(mul2(f2(ir[0]), pir[0]), pw[0]), go = mul2(mul2(pir[0], pir[0]), f2(qneg[0]));
        const float2 be = mul2(Sp[0], gi);
        aN[0] = fma2(be, px[0], aN[0]); aN[1] = fma2(be, py[0], aN[1]); aN[2] = fma2(be, pz[0], aN[2]);
        aN[3] = fma2(cin[0], gi, aN[3]);
        // to b_{i+t}, b_{i+t+8}; here from a_{i-t}, a_{i-t-8}
        const float2 ao = mul2(cout[0], go), bo = mul2(Sp[0], go);
        const int s1 = (i - t) & 15, s2 = (i - t + 8) & 15;
        const float2 ra = f2(__shfl_sync(M, ao.x, s1, 16), __shfl_sync(M, ao.y, s2, 16));
        const float2 rb = f2(__shfl_sync(M, bo.x, s1, 16), __shfl_sync(M, bo.y, s2, 16));
        const float4 c0 = PC[2 * s1];
        const float2 cz = *reinterpret_cast<const float2*>(&PC[2 * s1 + 1]);
        bN[0] = fma2(rb, f2(c0.x, c0.y), bN[0]); bN[1] = fma2(rb, f2(c0.z, c0.w), bN[1]);
        bN[2] = fma2(rb, cz, bN[2]);
        bN[3] = add2(ra, bN[3]);
      }
      {
        const float2 gab = mul2(irab, pir[1]), go2 = mul2(iro1, iro1);
        const float2 gm = mul2(sel2(me_inner, gab, go2), pw[1]);  // at my end, with the partner's weight
        const float2 be = mul2(Sp[1], gm);
        cN[0] = fma2(be, px[1], cN[0]); cN[1] = fma2(be, py[1], cN[1]); cN[2] = fma2(be, pz[1], cN[2]);
        cN[3] = fma2(sel2(me_inner, cin[1], cout[1]), gm, cN[3]);
        if (t < 7) {  // (at t = 7 both lanes of a pair took it)
          const float2 gp = mul2(sel2(me_inner, go2, gab), w);
          const float2 ao = mul2(sel2(me_inner, cout[1], cin[1]), gp), bo = mul2(Sp[1], gp);
          const int s1 = (i - t - 1) & 15;
          const float2 ra = f2(__shfl_sync(M, ao.x, s1, 16), __shfl_sync(M, ao.y, s1, 16));
          const float2 rb = f2(__shfl_sync(M, bo.x, s1, 16), __shfl_sync(M, bo.y, s1, 16));
          const float4 c0 = PA[3 * s1];
          const float2 cz = *reinterpret_cast<const float2*>(&PA[3 * s1 + 1]);
          cN[0] = fma2(rb, f2(c0.x, c0.y), cN[0]); cN[1] = fma2(rb, f2(c0.z, c0.w), cN[1]);
          cN[2] = fma2(rb, cz, cN[2]);
          cN[3] = add2(ra, cN[3]);
        }
      }
    }
    const float pf = a.pf_t;
    const float ala = cN[3].x + (aN[3].x + aN[3].y), alb = cN[3].y + (bN[3].x + bN[3].y);
    E[0][0] = f2(pf * (cN[0].x + (aN[0].x + aN[0].y) + ala * ux.x), 0.f);
    E[0][1] = f2(pf * (cN[1].x + (aN[1].x + aN[1].y) + ala * uy.x), 0.f);
    E[0][2] = f2(pf * (cN[2].x + (aN[2].x + aN[2].y) + ala * uz.x), 0.f);
    E[1][0] = f2(pf * (cN[0].y + (bN[0].x + bN[0].y) + alb * ux.y), 0.f);
    E[1][1] = f2(pf * (cN[1].y + (bN[1].x + bN[1].y) + alb * uy.y), 0.f);
    E[1][2] = f2(pf * (cN[2].y + (bN[2].x + bN[2].y) + alb * uz.y), 0.f);
  }

  // phase 1: the tiles' expansion coefficients (as in field_tile), in place of the
  // copied carries. Component e goes to word e + L (2 e for m = 0) of its run of complex
  // coefficients: a warp's stores, and the gathers of phase 2 for consecutive l, are
  // free of bank conflicts.
  copy_wait();
  __syncwarp();
  {
    const float2* gb = reinterpret_cast<const float2*>(a.gbase + g * NC);
    const uint16_t* ctab = g_comp + comp_tab_off(L);
    const float mpf = a.mpf, mpfr = a.mpfr;
    constexpr int NIT = (NC / 2 + 31) / 32;
    float2 v[2][NIT];
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      const int e = lane + 32 * it;
      if (e < NC / 2) {
        const uint16_t cr = ctab[e];
        const int l = cr & 0xff;
        const float rl = a.rhol[l];
        const float2 gv = gb[e];
        float im = a.f[l] * a.tot[2 * e + 1];
        if ((cr >> 8) & 1) im -= drive_of(a, l);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const float2 c = *reinterpret_cast<const float2*>(sc0 + t * SCW + 2 * e);
          v[t][it] = f2((rl * (gv.x + c.x) - im) * mpf, rl * (gv.y + c.y) * mpfr);
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
      const int e = lane + 32 * it;
      if (e < NC / 2) {
        const int o = e < L ? 2 * e : e + L;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          sc0[t * SCW + o] = v[t][it].x;
          sc0[t * SCW + 2 * pair_run(L) + o] = v[t][it].y;
          if (e < L) sc0[t * SCW + o + 1] = sc0[t * SCW + 2 * pair_run(L) + o + 1] = 0.f;
        }
      }
    }
    if (lane < 4) sc0[(lane >> 1) * SCW + 4 * pair_run(L) + (lane & 1)] = 0.f;
  }
  __syncwarp();

  // phase 2: the records k0 .. k1 - 1 of both tiles: per (l, m) the gradient's
  // factors of the multipole and of the local harmonic side by side,
  // (x, y, z of the real part), (x, y, z of the imaginary part)
  auto build = [&](int k0, int k1) {
    __syncwarp();
    constexpr int NB = (pair_most(L) + 31) / 32;
#pragma unroll 1
    for (int it = 0; it < NB; ++it) {
      const int k = k0 + lane + 32 * it;
      if (k < k1) {
        const PairSrc src = g_psrc[rec_off(L) + k];
        const float4 fac[2] = {g_pfac[0][rec_off(L) + k], g_pfac[1][rec_off(L) + k]};
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const float2* sc = reinterpret_cast<const float2*>(sc0 + t * SCW);
          float v[2][6];
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            const float2 c1 = sc[src.i[3 * s]], c2 = sc[src.i[3 * s + 1]], c0 = sc[src.i[3 * s + 2]];
            const float s1r = fac[s].x, s1i = fac[s].y, s2 = fac[s].z, sz = fac[s].w;
            v[s][0] = s1r * c1.x + s2 * c2.x;
            v[s][1] = s2 * c2.y - s1i * c1.y;
            v[s][2] = sz * c0.x;
            v[s][3] = s1i * c1.y + s2 * c2.y;
            v[s][4] = s1r * c1.x - s2 * c2.x;
            v[s][5] = sz * c0.y;
          }
          float4* o = rec0 + t * SR + 3 * (k - k0);
          o[0] = make_float4(v[0][0], v[1][0], v[0][1], v[1][1]);
          o[1] = make_float4(v[0][2], v[1][2], v[0][3], v[1][3]);
          o[2] = make_float4(v[0][4], v[1][4], v[0][5], v[1][5]);
        }
      }
    }
    __syncwarp();
  };
  const float4* const rec = rec0 + h * SR;

  // phase 3: the far field. Multipole and local harmonics share the recurrence's
  // coefficients, so one instruction advances both (first half: Is(x), second:
  // Rs(x / r_out), whose factors past its degrees are zero): column m is
  // (dr + i di) times the real p_l with p_{l+1} = an zz p_l - ww p_{l-1}, and the six
  // sums over l of a column are multiplied by its diagonal once.
  {
    float2 zz[2], ww[2], cx[2], cy[2], dr[2], di[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float ri = a.rho_inv, ir2 = 1.f / r2[p];
      zz[p] = f2(Z[p] * ir2, Z[p] * ri);
      ww[p] = f2(-ir2, -(r2[p] * ri * ri));
      cx[p] = f2(X[p] * ir2, X[p] * ri);
      cy[p] = f2(Y[p] * ir2, Y[p] * ri);
      dr[p] = f2(ir[p], 1.f);
      di[p] = f2(0.f);
    }
#pragma unroll
    for (int q = 0; q < pair_nchunk(L); ++q) {
      const int m0 = pair_chunk(L, q), m1 = pair_chunk(L, q + 1), k0 = offP(L, m0);
      build(k0, offP(L, m1));
      if (m0 == 0) {  // the real column m = 0
        float2 p1[2] = {dr[0], dr[1]}, p0[2] = {f2(0.f), f2(0.f)};
        auto add = [&](int l) {
          const float4 r0 = rec[3 * l];
          const float2 rz = *reinterpret_cast<const float2*>(&rec[3 * l + 1]);
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            E[p][0] = fma2(f2(r0.x, r0.y), p1[p], E[p][0]);
            E[p][1] = fma2(f2(r0.z, r0.w), p1[p], E[p][1]);
            E[p][2] = fma2(rz, p1[p], E[p][2]);
          }
        };
        add(0);
#pragma unroll 2
        for (int l = 1; l <= L + 1; ++l) {  // (unrolled whole, its products fill the registers)
          const float2 c = c_an2[l];
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const float2 pn = fma2(mul2(c, zz[p]), p1[p], mul2(ww[p], p0[p]));
            p0[p] = p1[p]; p1[p] = pn;
          }
          add(l);
        }
      }
#pragma unroll 1
      for (int m = m0 > 1 ? m0 : 1; m < m1; ++m) {
        const float2 dg = f2(tb.dg[m]);
        const float4* rc = rec + 3 * (offP(L, m) - k0);
        const float2* an = c_an2 + m * kTabL;
        float2 p1[2], p0[2], S[2][3], T[2][3];
        {
          const float4 r0 = rc[0], r1 = rc[1], r2_ = rc[2];
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const float2 ex = mul2(dg, cx[p]), ey = mul2(dg, cy[p]);
            const float2 nr = fma2(ex, dr[p], neg2(mul2(ey, di[p]))), ni = fma2(ex, di[p], mul2(ey, dr[p]));
            dr[p] = nr; di[p] = ni;
            p1[p] = f2(1.f); p0[p] = f2(0.f);
            S[p][0] = f2(r0.x, r0.y); S[p][1] = f2(r0.z, r0.w); S[p][2] = f2(r1.x, r1.y);
            T[p][0] = f2(r1.z, r1.w); T[p][1] = f2(r2_.x, r2_.y); T[p][2] = f2(r2_.z, r2_.w);
          }
        }
#pragma unroll 4
        for (int jj = 1; jj <= L + 1 - m; ++jj) {
          const float2 c = an[jj];
          const float4 r0 = rc[3 * jj], r1 = rc[3 * jj + 1], r2_ = rc[3 * jj + 2];
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            const float2 pn = fma2(mul2(c, zz[p]), p1[p], mul2(ww[p], p0[p]));
            p0[p] = p1[p]; p1[p] = pn;
            S[p][0] = fma2(f2(r0.x, r0.y), pn, S[p][0]);
            S[p][1] = fma2(f2(r0.z, r0.w), pn, S[p][1]);
            S[p][2] = fma2(f2(r1.x, r1.y), pn, S[p][2]);
            T[p][0] = fma2(f2(r1.z, r1.w), pn, T[p][0]);
            T[p][1] = fma2(f2(r2_.x, r2_.y), pn, T[p][1]);
            T[p][2] = fma2(f2(r2_.z, r2_.w), pn, T[p][2]);
          }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
          for (int k = 0; k < 3; ++k) E[p][k] = fma2(dr[p], S[p][k], fma2(di[p], T[p][k], E[p][k]));
      }
    }
  }

  double qmob[2] = {0.0, 0.0};
  if (a.species) {
    const double qa = -double(qneg[0]), qb = -double(qneg[1]);  // 0 in an empty place
    double ia = qa, ib = qb;
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
      const double ta = __shfl_up_sync(0xffffffffu, ia, d, 16), tb2 = __shfl_up_sync(0xffffffffu, ib, d, 16);
      if (i >= d) { ia += ta; ib += tb2; }
    }
    const double before = a.qgbase[g] + (valid[0] ? a.qpfx[tile] : 0.0);
    qmob[0] = before + (ia - qa);
    qmob[1] = before + __shfl_sync(0xffffffffu, ia, 15, 16) + (ib - qb);
  }
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    // the particle again (kept in shared memory meanwhile)
    const int o = 32 * h + 16 * p + i;
    const int64_t jp = tile * 32 + 16 * p + i;
    const bool ok = jp < a.n;
    const float x = vel[256 + o], y = vel[320 + o], z = vel[384 + o];
    const uint32_t* id = reinterpret_cast<const uint32_t*>(vel + 192 + o);
    const bool ion = a.species && ok && *id >= a.n_e;
    const float rr = x * x + y * y + z * z;
    field_finish<float, L>(a, jp, ok, ion, ok ? (ion ? -a.q_ion : 1.f) : 0.f, x, y, z, vel[o], vel[64 + o], vel[128 + o],
                           rr, 1.f / rr, rsqrtf(rr), E[p][0].x + E[p][0].y, E[p][1].x + E[p][1].y,
                           E[p][2].x + E[p][2].y, qmob[p], q_s, id);
  }
}

// 128 registers (4 CTAs of 128 threads): with 96 the near field spills and the
// kernel is slower (l_max = 16: 0.553 against 0.470 ms).
template <int L>
__global__ void __launch_bounds__(kPairMaxWarps * 32, 4) k_field_pair(FieldArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chain_wait();
  const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  field_pair<L>(a, smem_raw, warp, int64_t(gridDim.x - 1 - blockIdx.x) * wpb + warp);
}

// Batched: CTA b takes the pairs of tiles from items[b].y on of instance items[b].x.
template <int L>
__global__ void __launch_bounds__(kPairMaxWarps * 32, 4) k_field_pair_batch(const FieldArgs<float>* __restrict__ args,
                                                                          const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FieldArgs<float> sa;
  const int2 it = items[blockIdx.x];
  copy_args(args + it.x, &sa);
  __syncthreads();
  field_pair<L>(sa, smem_raw, threadIdx.x >> 5, int64_t(it.y) + (threadIdx.x >> 5));
}

// ----------------------------------------------------------------------------
// Field kernel of FP64 instances: one CTA of four warps per tile. FP64 runs at 1/64
// of the FP32 rate (half a lane per clock and scheduler), so the operation count is
// what bounds it, and a tile held by one warp keeps three of an SM's four FP64 pipes
// idle when there are few tiles. Warp w takes every fourth column of the far field
// and every fourth round of the near field; the partial fields are added in a fixed
// order. Operations per particle at l_max = 16: 2600 far + 2200 near (field_tile: 3300
// + 2900): multipole and local part share the angular recurrence and the diagonal
// (powers of r from a table in shared memory, whose pipe is idle), the pair sums run
// by Clenshaw's recurrence. Field ms, field_tile (its best CTA size) -> this: l_max = 8,
// N = 3001: 0.092 -> 0.038, N = 20000: 0.130 -> 0.115 (5 tiles on the fullest SM, 4.1 on
// average), N = 40000: 0.266 -> 0.194; l_max = 12, N = 60000: 0.486 -> 0.415; l_max = 16,
// N = 250001: 2.49 -> 2.28; l_max = 2, N = 1e6: 1.79 -> 1.54.
// ----------------------------------------------------------------------------
__host__ __device__ constexpr size_t team_smem(int L) {
  return sizeof(double) * (size_t(12) * nP(L) + 32 * (2 * L + 2) + 32 * 6 + kTeam * 3 * 32 + 2 * (2 * pair_run(L) + 1));
}

// The pair sums of pair_sums, for one pair in FP64.
template <int L>
__device__ __forceinline__ void pair_sums_f64(double x1, double y2, double& S0, double& S1, double& S2) {
  double b1 = leg_c(L), b2 = 0.0, d1 = L * leg_c(L), d2 = 0.0, e1 = 0.0, e2 = 0.0;
#pragma unroll
  for (int l = L - 1; l >= 0; --l) {
    const double G = -leg_g(l + 1) * y2;
    double nb = l > 0 ? leg_c(l) : 0.0, nd = l > 0 ? l * leg_c(l) : 0.0, ne = b1;
    if (l < L - 1) {
      nb = l > 0 ? fma(G, b2, nb) : G * b2;
      nd = l > 0 ? fma(G, d2, nd) : G * d2;
      if (l < L - 2) ne = fma(G, e2, ne);
      ne = fma(x1, e1, ne);
    }
    nb = l == 0 && L == 1 ? x1 * b1 : fma(x1, b1, nb);
    nd = l == 0 && L == 1 ? x1 * d1 : fma(x1, d1, nd);
    b2 = b1; b1 = nb; d2 = d1; d1 = nd; e2 = e1; e1 = ne;
  }
  S0 = b1; S1 = d1; S2 = e1;
}

template <int L>
__device__ __forceinline__ void field_team(const FieldArgs<double>& a, unsigned char* smem_raw, int64_t tile) {
  constexpr int NC = 2 * ncomp(L), NP = nP(L), RUN = pair_run(L);
  const Tables<double>& tb = tab<double>();
  const int lane = int(lane_id()), warp = threadIdx.x >> 5;
  double* const rec = reinterpret_cast<double*>(smem_raw);       // [NP][12]
  double* const uI = rec + 12 * NP;                              // [L + 2][32]: r^-(l+1)
  double* const uR = uI + 32 * (L + 2);                          // [L][32]: (r / r_out)^l
  double2* const pd = reinterpret_cast<double2*>(uR + 32 * L);   // [32][3]: (ex, ey), (ez, r), (1/r, -q)
  double* const part = reinterpret_cast<double*>(pd + 32 * 3);   // [kTeam][3][32]
  double2* const sc = reinterpret_cast<double2*>(part + kTeam * 3 * 32);
  const int64_t g = tile / kTilesPerGroup;
  const int64_t j = tile * 32 + lane;
  const bool valid = j < a.n;
  // warp 0 prepares the particles and the powers of r (once per tile: a reciprocal
  // root alone is some 20 FP64 operations), the others form the coefficients
  if (warp == 0) {
    const double X = valid ? a.x[j] : a.r_out, Y = valid ? a.y[j] : 0.0, Z = valid ? a.z[j] : 0.0;
    const double r2 = X * X + Y * Y + Z * Z, ir = rsqrt(r2), rk = r2 * ir;
    pd[3 * lane] = make_double2(X * ir, Y * ir);
    pd[3 * lane + 1] = make_double2(Z * ir, rk);
    pd[3 * lane + 2] = make_double2(ir, valid ? (a.species && a.id[j] >= a.n_e ? -a.q_ion : 1.0) : 0.0);
    const double q = rk * a.rho_inv;
    double u = ir, w = 1.0;
#pragma unroll 2
    for (int l = 0; l <= L + 1; ++l) {
      uI[32 * l + lane] = u;
      u *= ir;
      if (l < L) uR[32 * l + lane] = w;
      w *= q;
    }
  } else {
    // phase 1: the tile's expansion coefficients (as in field_tile)
    const double2* pt = reinterpret_cast<const double2*>(a.pfx + tile * NC);
    const double2* gb = reinterpret_cast<const double2*>(a.gbase + g * NC);
    const uint16_t* ctab = g_comp + comp_tab_off(L);
    double* const s0 = reinterpret_cast<double*>(sc);
    for (int e = threadIdx.x - 32; e < NC / 2; e += (kTeam - 1) * 32) {
      const uint16_t cr = ctab[e];
      const int l = cr & 0xff;
      const double rl = a.rhol[l];
      const double2 ab = pt[e], gv = gb[e];
      double cI = rl * (gv.x + ab.x) - a.f[l] * a.tot[2 * e + 1];
      if ((cr >> 8) & 1) cI += drive_of(a, l);
      const int o = e < L ? 2 * e : e + L;
      s0[o] = cI * a.mpf;
      s0[2 * RUN + o] = rl * (gv.y + ab.y) * a.mpfr;
      if (e < L) s0[o + 1] = s0[2 * RUN + o + 1] = 0.0;
    }
    if (threadIdx.x == 32) sc[2 * RUN] = make_double2(0.0, 0.0);
  }
  __syncthreads();
  const double2 d0 = pd[3 * lane], d1 = pd[3 * lane + 1], d2 = pd[3 * lane + 2];
  const double ex = d0.x, ey = d0.y, ez = d1.x, rk = d1.y, ir = d2.x, qneg = d2.y;
  // phase 2: the gradient factors per (l, m): real x, y, z, imaginary x, y, z of the
  // multipole and of the local entry
  for (int k = threadIdx.x; k < NP; k += kTeam * 32) {
    const PairSrc src = g_psrc[rec_off(L) + k];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const TeamFac f = g_tfac[s][rec_off(L) + k];
      const double2 c1 = sc[src.i[3 * s]], c2 = sc[src.i[3 * s + 1]], c0 = sc[src.i[3 * s + 2]];
      double2* o = reinterpret_cast<double2*>(rec + 12 * k + 6 * s);
      o[0] = make_double2(f.s1r * c1.x + f.s2 * c2.x, f.s2 * c2.y - f.s1i * c1.y);
      o[1] = make_double2(f.sz * c0.x, f.s1i * c1.y + f.s2 * c2.y);
      o[2] = make_double2(f.s1r * c1.x - f.s2 * c2.x, f.sz * c0.y);
    }
  }
  // near field: rounds s = warp + 1, warp + 5, ... of the ring of 32 (as field_tile's,
  // with the factors of field_pair); round 16 is taken by both lanes of a pair
  double Nx = 0.0, Ny = 0.0, Nz = 0.0, Na = 0.0;
#pragma unroll 1
  for (int s = warp + 1; s <= 16; s += kTeam) {
    const int src = (lane + s) & 31;
    const bool me_inner = lane < src;
    const double2 p0 = pd[3 * src], p1 = pd[3 * src + 1], p2 = pd[3 * src + 2];
    const double u = ex * p0.x + ey * p0.y + ez * p1.x;
    const double iro = me_inner ? p2.x : ir, sr = (me_inner ? rk : p1.y) * iro;
    double S0, S1, S2;
    pair_sums_f64<L>(sr * u, sr * sr, S0, S1, S2);
    const double Sp = S2 * sr, uS = u * Sp;
    const double cin = S1 - uS, cout = -(S0 + S1 + uS);
    const double gab = ir * p2.x, go2 = iro * iro;
    const double gm = (me_inner ? gab : go2) * p2.y, be = Sp * gm;
    Nx = fma(be, p0.x, Nx); Ny = fma(be, p0.y, Ny); Nz = fma(be, p1.x, Nz);
    Na = fma(me_inner ? cin : cout, gm, Na);
    if (s < 16) {
      const double gp = (me_inner ? go2 : gab) * qneg;
      const double ao = (me_inner ? cout : cin) * gp, bo = Sp * gp;
      const int from = (lane - s) & 31;
      const double ra = __shfl_sync(0xffffffffu, ao, from), rb = __shfl_sync(0xffffffffu, bo, from);
      const double2 c0 = pd[3 * from], c1 = pd[3 * from + 1];
      Nx = fma(rb, c0.x, Nx); Ny = fma(rb, c0.y, Ny); Nz = fma(rb, c1.x, Nz);
      Na += ra;
    }
  }
  double Ex = a.pf_t * (Nx + Na * ex), Ey = a.pf_t * (Ny + Na * ey), Ez = a.pf_t * (Nz + Na * ez);
  __syncthreads();
  // phase 3: far-field columns m = warp, warp + 4, ...: (ex + i ey)^m times the sums over
  // l of the real p_l, p_{l+1} = an cos(t) p_l - p_{l-1}, with both parts' factors and powers
  {
    double dr = 1.0, di = 0.0;
    for (int k = 0; k < warp; ++k) {
      const double t = dr * ex - di * ey;
      di = dr * ey + di * ex;
      dr = t;
    }
    const double q2r = ex * ex - ey * ey, q2i = 2.0 * ex * ey;
    const double q4r = q2r * q2r - q2i * q2i, q4i = 2.0 * q2r * q2i;
#pragma unroll 1
    for (int m = warp; m <= L + 1; m += kTeam) {
      double p1 = 1.0, p0 = 0.0;
      double Sx = 0.0, Sy = 0.0, Sz = 0.0, Tx = 0.0, Ty = 0.0, Tz = 0.0;
      const double2* rc = reinterpret_cast<const double2*>(rec + 12 * offP(L, m));
      auto step = [&](int l) {
        if (l > m) {
          const double pn = fma(tb.an[l * kTabL + m] * ez, p1, -p0);
          p0 = p1; p1 = pn;
        }
      };
      auto add = [&](const double2* c, double p) {
        const double2 c0 = c[0], c1 = c[1];
        Sx = fma(c0.x, p, Sx); Sy = fma(c0.y, p, Sy); Sz = fma(c1.x, p, Sz);
        if (m > 0) {
          const double2 c2 = c[2];
          Tx = fma(c1.y, p, Tx); Ty = fma(c2.x, p, Ty); Tz = fma(c2.y, p, Tz);
        }
      };
      int l = m;
#pragma unroll 2
      for (; l <= L - 1; ++l, rc += 6) {
        step(l);
        add(rc, p1 * uI[32 * l + lane]);
        add(rc + 3, p1 * uR[32 * l + lane]);
      }
      for (; l <= L + 1; ++l, rc += 6) {
        step(l);
        add(rc, p1 * uI[32 * l + lane]);
      }
      Ex = fma(dr, Sx, fma(di, Tx, Ex)); Ey = fma(dr, Sy, fma(di, Ty, Ey)); Ez = fma(dr, Sz, fma(di, Tz, Ez));
      const double t = dr * q4r - di * q4i;
      di = dr * q4i + di * q4r;
      dr = t;
    }
  }
  part[96 * warp + lane] = Ex;
  part[96 * warp + 32 + lane] = Ey;
  part[96 * warp + 64 + lane] = Ez;
  __syncthreads();
  if (warp != kTeam - 1) return;  // the warp with the shortest columns goes on
  Ex = Ey = Ez = 0.0;
#pragma unroll
  for (int w = 0; w < kTeam; ++w) {
    Ex += part[96 * w + lane]; Ey += part[96 * w + 32 + lane]; Ez += part[96 * w + 64 + lane];
  }
  double qmob = 0.0;
  if (a.species) {
    const double qc = -qneg;
    double incl = qc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    qmob = a.qgbase[g] + a.qpfx[tile] + (incl - qc);
  }
  const bool push = a.mode == 0 && valid;
  const double VX = push ? a.vx[j] : 0.0, VY = push ? a.vy[j] : 0.0, VZ = push ? a.vz[j] : 0.0;
  const double X = valid ? a.x[j] : a.r_out, Y = valid ? a.y[j] : 0.0, Z = valid ? a.z[j] : 0.0;
  field_finish<double, L>(a, j, valid, valid && qneg != 1.0, qneg, X, Y, Z, VX, VY, VZ, rk * rk, ir * ir, ir, Ex, Ey, Ez, qmob,
                          a.q_s + a.st->qs_acc, a.id + j);
}

template <int L>
__global__ void __launch_bounds__(kTeam * 32) k_field_team(FieldArgs<double> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chain_wait();
  field_team<L>(a, smem_raw, int64_t(gridDim.x) - 1 - blockIdx.x);
}
template <int L>
__global__ void __launch_bounds__(kTeam * 32) k_field_team_batch(const FieldArgs<double>* __restrict__ args,
                                                               const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FieldArgs<double> sa;
  const int2 it = items[blockIdx.x];
  copy_args(args + it.x, &sa);
  __syncthreads();
  field_team<L>(sa, smem_raw, it.y);
}

// Register budget: in FP32, at least 3 CTAs of 256 threads per SM (80
// registers): ptxas otherwise settles at 64 with spills in the far-field
// loops; FP64 keeps its ~124.
template <class T>
__host__ __device__ constexpr int field_min_blocks() { return sizeof(T) == 4 ? 3 : 1; }

template <class T, int L>
__global__ void __launch_bounds__(256, field_min_blocks<T>()) k_field(FieldArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chain_wait();
  const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  // tiles in decreasing order: the particle rows written last (still in L2) first
  field_tile<T, L, 0>(a, smem_raw, warp, wpb, int64_t(gridDim.x - 1 - blockIdx.x) * wpb + warp);
}

// The same for contexts of img_in_tile (at most kImgInTileMaxN particles), four image pairs at a
// time: these launches leave one warp to an SM, whose recurrences would wait for each other, and
// registers to spare (in k_field, capped for its occupancy, the code alone cost 2 % by spills).
// Field of N = 1000, l_max = 8: 0.033 ms with one pair at a time and a division per pair and
// degree, 0.0227 so; the call without allocations 82.9 -> 71.9 us.
constexpr int kImgPairs = 4;
template <int L>
__global__ void __launch_bounds__(256, 1) k_field_small(FieldArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  chain_wait();
  const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  field_tile<float, L, kImgPairs>(a, smem_raw, warp, wpb, int64_t(blockIdx.x) * wpb + warp);
}

// Batched field: the instances of one degree and precision in one launch. CTA
// b takes the tiles items[b].y .. items[b].y + wpb - 1 of instance items[b].x,
// whose arguments args[items[b].x] are first copied to shared memory (a warp
// past its instance's last tile returns at once, as in the single launch).
template <class T, int L>
__global__ void __launch_bounds__(256, field_min_blocks<T>()) k_field_batch(const FieldArgs<T>* __restrict__ args,
                                                     const int2* __restrict__ items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ FieldArgs<T> sa;
  const int2 it = items[blockIdx.x];
  copy_args(args + it.x, &sa);
  __syncthreads();
  const int warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  field_tile<T, L, sizeof(T) == 4 ? 1 : 0>(sa, smem_raw, warp, wpb, int64_t(it.y) + warp);
}

}  // namespace imrp
