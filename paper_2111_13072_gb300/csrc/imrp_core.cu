// Degree-independent kernels of the IMRP hot path: the radius radix sort, state
// reorder, key generation, loading, the FP64 scans of the tile moments, the
// per-step finalize (drive u_asy and the Q_diff tally), and the spectrum sums.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "imrp_internal.h"

namespace imrp {

// ============================================================================
// Global passes (arrays too large for the bucket sort below): a stable LSD radix
// sort of 8-bit digits. Each CTA owns kSortTile = 2048 consecutive keys in a
// striped layout (item i of thread t is key base + i*256 + t), which keeps the
// slot order (item, warp, lane) equal to the key order, so the local ranks below
// are stable; hist holds 256 rows of nblk block counts.
// ============================================================================
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const uint32_t* __restrict__ keys,
                                                           int64_t n, int shift, int64_t nblk,
                                                           uint32_t* __restrict__ hist) {
  chain_wait();
  constexpr int ND = 256;
  __shared__ uint32_t h[ND];
  for (int d = threadIdx.x; d < ND; d += kSortThreads) h[d] = 0;
  __syncthreads();
  const int64_t base = int64_t(blockIdx.x) * kSortTile;
  const int nvalid = n - base < kSortTile ? int(n - base) : kSortTile;
  const unsigned lane = threadIdx.x & 31;
  uint32_t k[kSortItems];
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const int o = i * kSortThreads + int(threadIdx.x);
    k[i] = o < nvalid ? keys[base + o] : 0u;
  }
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    // a warp holds 32 consecutive keys: when they share the digit (nearly
    // sorted input), one atomic adds all 32
    const bool ok = i * kSortThreads + int(threadIdx.x) < nvalid;
    const unsigned d = (k[i] >> shift) & unsigned(ND - 1);
    const unsigned d0 = __shfl_sync(0xffffffffu, d, 0);
    if (__all_sync(0xffffffffu, ok && d == d0)) {
      if (lane == 0) atomicAdd(&h[d0], 32u);
    } else if (ok) {
      atomicAdd(&h[d], 1u);
    }
  }
  __syncthreads();
  for (int d = threadIdx.x; d < ND; d += kSortThreads) hist[int64_t(d) * nblk + blockIdx.x] = h[d];
}

// Exclusive prefix over the kSortThreads threads of a CTA of the per-thread
// values v (warp shuffles, then the warp sums through wsum); *total gets the
// sum over the CTA. All threads call it; the caller separates two uses of wsum
// by a barrier.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* wsum, uint32_t* total = nullptr) {
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= unsigned(o)) s += x;
  }
  if (lane == 31) wsum[warp] = s;
  __syncthreads();
  uint32_t woff = 0, tot = 0;
#pragma unroll
  for (unsigned w = 0; w < kSortThreads / 32; ++w) {
    const uint32_t x = wsum[w];
    woff += w < warp ? x : 0u;
    tot += x;
  }
  if (total) *total = tot;
  return woff + s - v;
}

// Exclusive scan of one digit's row hist[d][0..nblk) in place; the row total
// goes to rowtot[d]. One CTA per digit.
__global__ void __launch_bounds__(kSortThreads) k_sort_rowscan(uint32_t* __restrict__ hist, int64_t nblk,
                                                              uint32_t* __restrict__ rowtot) {
  chain_wait();
  constexpr int R = 8;  // consecutive entries per thread, loaded together
  __shared__ uint32_t wsum[kSortThreads / 32];
  uint32_t* row = hist + int64_t(blockIdx.x) * nblk;
  uint32_t carry = 0;
  for (int64_t b0 = 0; b0 < nblk; b0 += int64_t(kSortThreads) * R) {
    const int64_t i0 = b0 + int64_t(R) * threadIdx.x;
    uint32_t v[R], sum = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = i0 + r < nblk ? row[i0 + r] : 0u;
      sum += v[r];
    }
    uint32_t tot;
    uint32_t run = carry + block_excl_scan(sum, wsum, &tot);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (i0 + r < nblk) row[i0 + r] = run;
      run += v[r];
    }
    carry += tot;
    __syncthreads();  // wsum reuse
  }
  if (threadIdx.x == 0) rowtot[blockIdx.x] = carry;
}

// Lanes of the warp whose digit equals this lane's (bits BITS of d), among
// the lanes with ok set: one ballot per digit bit.
template <int BITS>
__device__ __forceinline__ unsigned digit_peers(unsigned d, bool ok) {
  unsigned p = __ballot_sync(0xffffffffu, ok);
#pragma unroll
  for (int b = 0; b < BITS; ++b) {
    const unsigned m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
    p &= ((d >> b) & 1u) ? m : ~m;
  }
  return p;
}

// Scatter of one pass. Warp w of the block owns the keys base + 256 w ..
// base + 256 w + 255 (item i of lane l is key base + 256 w + 32 i + l), so the
// order (warp, item, lane) is the key order. The items of a warp are ranked
// one after the other against the warp's running digit counts whist[w][d];
// a key's block-local position is then (start of its digit in the block) +
// (keys of that digit in earlier warps) + (its rank in its warp): stable.
// The block's keys and slots are staged in shared memory in that order, so
// that consecutive threads write consecutive positions of each digit's run
// in the output (coalesced even when the digits are uniformly spread). Thread
// t owns digit t in the per-digit steps. About 22 KB of shared memory and at most
// 36 registers per thread (7 blocks per SM). Ranking by __match_any_sync (faster
// here than ballots).
__global__ void __launch_bounds__(kSortThreads, 7) k_sort_scatter(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, int64_t n, int shift, int64_t nblk,
    const uint32_t* __restrict__ hist, const uint32_t* __restrict__ rowtot) {
  chain_wait();
  constexpr int kWarps = kSortThreads / 32;
  constexpr int ND = 256, DPT = ND / kSortThreads;
  static_assert(kSortItems * 32 <= 256 && kSortTile <= 65535, "per-warp counts fit 16 bits");
  __shared__ __align__(16) uint16_t whist[kWarps][ND];
  __shared__ __align__(16) uint32_t sk[kSortTile];
  __shared__ __align__(16) uint32_t sv[kSortTile];
  __shared__ uint32_t dbase[ND];   // global start of digit d for this block
  __shared__ uint32_t lstart[ND];  // block-local start of digit d
  __shared__ uint32_t wsum[kWarps];
  const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
  {
    uint4* z = reinterpret_cast<uint4*>(&whist[0][0]);
    for (int k = t; k < kWarps * ND * 2 / 16; k += kSortThreads) z[k] = make_uint4(0u, 0u, 0u, 0u);
  }
  // exclusive scan of the digit totals -> global start of each digit
  {
    uint32_t c[DPT], sum = 0;
#pragma unroll
    for (int k = 0; k < DPT; ++k) {
      c[k] = rowtot[DPT * t + k];
      sum += c[k];
    }
    uint32_t off = block_excl_scan(sum, wsum);
#pragma unroll
    for (int k = 0; k < DPT; ++k) {
      const unsigned d = DPT * t + k;
      dbase[d] = off + hist[int64_t(d) * nblk + blockIdx.x];
      off += c[k];
    }
  }
  const int64_t base = int64_t(blockIdx.x) * kSortTile;
  const int64_t wbase = base + int64_t(warp) * (32 * kSortItems);
  const unsigned lt = (1u << lane) - 1u;
  uint32_t key[kSortItems];
  uint32_t wrank[(kSortItems + 3) / 4] = {};  // rank in the warp (< 256), one byte per item
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const int64_t idx = wbase + 32 * i + lane;
    key[i] = idx < n ? kin[idx] : 0u;
  }
  __syncthreads();  // whist zeroed, wsum consumed
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const bool ok = wbase + 32 * i + lane < n;
    const unsigned d = ok ? ((key[i] >> shift) & unsigned(ND - 1)) : unsigned(ND);
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const unsigned before = ok ? unsigned(whist[warp][d]) : 0u;
    wrank[i / 4] |= (before + __popc(peers & lt)) << (8 * (i % 4));
    __syncwarp();
    if (ok && lane == unsigned(__ffs(peers) - 1)) whist[warp][d] = uint16_t(before + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  // block count of each digit of this thread; whist[w][d] becomes the count in warps before w
  uint32_t total[DPT], tsum = 0;
#pragma unroll
  for (int k = 0; k < DPT; ++k) {
    const unsigned d = DPT * t + k;
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = whist[w][d];
      whist[w][d] = uint16_t(run);
      run += c;
    }
    total[k] = run;
    tsum += run;
  }
  // block-local digit starts: exclusive scan of the block counts over d
  {
    __syncthreads();  // wsum reuse
    uint32_t off = block_excl_scan(tsum, wsum);
#pragma unroll
    for (int k = 0; k < DPT; ++k) {
      lstart[DPT * t + k] = off;
      off += total[k];
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const int64_t idx = wbase + 32 * i + lane;
    if (idx < n) {
      const unsigned d = (key[i] >> shift) & unsigned(ND - 1);
      const uint32_t lpos = lstart[d] + whist[warp][d] + ((wrank[i / 4] >> (8 * (i % 4))) & 255u);
      sk[lpos] = key[i];
      sv[lpos] = vin[idx];
    }
  }
  __syncthreads();
  const int64_t nvalid = n - base < kSortTile ? n - base : kSortTile;
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const int p = i * kSortThreads + int(t);
    if (p < nvalid) {
      const uint32_t k = sk[p];
      const unsigned d = (k >> shift) & unsigned(ND - 1);
      const uint32_t g = dbase[d] + (uint32_t(p) - lstart[d]);
      kout[g] = k;
      vout[g] = sv[p];
    }
  }
}

// Stable byte pass of one CTA over a bucket in global memory (in L2; the CTA alone touches
// that range): the scan of the byte's digit counts, then the bucket in chunks of NT * kBsItems
// keys in order; each warp ranks its keys (item i of lane l is slot 32 i + l of its part of the
// chunk) against its running digit counts, the warps' counts are scanned per digit, and each
// key goes to (digit start) + (keys of that digit in earlier chunks and warps) + (its rank in
// its warp). A warp whose part of the chunk holds no keys, and items past the end, skip the
// ranking. The peers of a key in its warp come from one ballot per digit bit.
constexpr int kBsItems = 4;

template <int NT> struct BsShared {
  uint32_t cnt[256];                 // digit counts of this pass's byte
  uint32_t dst[256];                 // output place of the next key of digit d
  uint16_t whist[NT / 32][256];      // per-warp counts, then the counts of earlier warps
  uint32_t wsum[8];
};

// One pass over len (< 2^31) keys (slots 0 .. len-1 of ki/vi into ko/vo), digit =
// byte at `shift`, whose counts are in sh.cnt.
template <int NT>
__device__ __forceinline__ void bucket_pass(const uint32_t* ki, const uint32_t* vi, uint32_t* ko, uint32_t* vo, int len,
                                            int shift, BsShared<NT>& sh) {
  constexpr int kWarps = NT / 32, kChunk = NT * kBsItems;
  const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t c = 0, s1 = 0;
  if (t < 256) {
    c = sh.cnt[t];
    s1 = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, s1, o);
      if (lane >= unsigned(o)) s1 += x;
    }
    if (lane == 31) sh.wsum[warp] = s1;
  }
  __syncthreads();
  if (t < 256) {
    uint32_t off = 0;
    for (unsigned w = 0; w < warp; ++w) off += sh.wsum[w];
    sh.dst[t] = off + s1 - c;
  }
  for (int c0 = 0; c0 < len; c0 += kChunk) {
    for (int k = t; k < kWarps * 256; k += NT) (&sh.whist[0][0])[k] = 0;
    __syncthreads();
    const int wb = c0 + int(warp) * (32 * kBsItems);
    const int nv = len - wb;  // keys of this warp's range that exist (warp-uniform)
    uint32_t key[kBsItems], val[kBsItems];
    uint32_t wrank[(kBsItems + 1) / 2] = {};
    if (nv > 0) {
#pragma unroll
      for (int i = 0; i < kBsItems; ++i) {
        const int o = 32 * i + int(lane);
        key[i] = o < nv ? ki[wb + o] : 0u;
        val[i] = o < nv ? vi[wb + o] : 0u;
      }
#pragma unroll
      for (int i = 0; i < kBsItems; ++i) {
        if (32 * i >= nv) break;
        const bool ok = 32 * i + int(lane) < nv;
        const unsigned d = ok ? ((key[i] >> shift) & 255u) : 256u;
        const unsigned peers = digit_peers<8>(d, ok);
        const unsigned before = ok ? unsigned(sh.whist[warp][d]) : 0u;
        wrank[i / 2] |= (before + __popc(peers & lt)) << (16 * (i % 2));
        __syncwarp();
        if (ok && lane == unsigned(__ffs(peers) - 1)) sh.whist[warp][d] = uint16_t(before + __popc(peers));
        __syncwarp();
      }
    }
    __syncthreads();
    uint32_t total = 0;
    if (t < 256) {
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        const uint32_t x = sh.whist[w][t];
        sh.whist[w][t] = uint16_t(total);
        total += x;
      }
    }
    __syncthreads();
    if (nv > 0) {
#pragma unroll
      for (int i = 0; i < kBsItems; ++i) {
        if (32 * i >= nv) break;
        if (32 * i + int(lane) < nv) {
          const unsigned d = (key[i] >> shift) & 255u;
          const uint32_t g = sh.dst[d] + sh.whist[warp][d] + ((wrank[i / 2] >> (16 * (i % 2))) & 0xffffu);
          ko[g] = key[i];
          vo[g] = val[i];
        }
      }
    }
    __syncthreads();
    if (t < 256) sh.dst[t] += total;
  }
  __syncthreads();  // this pass's writes are visible to the CTA's next pass
}

// Counts of the byte at `shift` of keys[0 .. len) into cnt (loads in flight together).
template <int NT>
__device__ __forceinline__ void count_byte(const uint32_t* keys, int64_t len, int shift, uint32_t* cnt) {
  for (int64_t i0 = 0; i0 < len; i0 += int64_t(NT) * kBsItems) {
    uint32_t k[kBsItems];
#pragma unroll
    for (int i = 0; i < kBsItems; ++i) {
      const int64_t idx = i0 + int64_t(i) * NT + threadIdx.x;
      k[i] = idx < len ? keys[idx] : 0u;
    }
#pragma unroll
    for (int i = 0; i < kBsItems; ++i) {
      const bool ok = i0 + int64_t(i) * NT + threadIdx.x < len;
      const unsigned d = (k[i] >> shift) & 255u, d0 = __shfl_sync(0xffffffffu, d, 0);
      if (__all_sync(0xffffffffu, ok && d == d0)) {  // 32 keys of one digit: one atomic
        if (threadIdx.x % 32 == 0) atomicAdd(&cnt[d0], 32u);
      } else if (ok) {
        atomicAdd(&cnt[d], 1u);
      }
    }
  }
}

// ---- bucket sort: top digit over the whole array, then each bucket in one CTA ----
// First pass: the keys' top digit (log2 nd bits, nd <= kSortDigits) over the whole array, in
// two kernels. k_sort_count adds up the digits (per CTA in shared memory, then one atomic per
// digit that occurs), and its last CTA to finish (an atomic ticket, no waiting) turns the totals
// into the buckets' starts; k_sort_spread reserves each digit's keys of a CTA with one atomic on
// the bucket's cursor and writes them there, in any order: the order within a bucket is settled
// by the comparisons of k_bucket_sort, so the result does not depend on the order of the atomics.
// In its scratch (SortState) the totals and the ticket are zero between sorts: whoever allocates it
// zeroes it in the order of the stream that sorts. Were they not, the cursors would lead out of the
// arrays: a place past the end is skipped, and a bucket that is no part of the array left out, with
// an error status that the next synchronising call returns.
// The stable pass (histogram matrix, row scan, ranked scatter; it serves the four global passes of
// very large arrays) took 7 + 6 + 20 us at N = 2e6; these two take 10 + 16, bound by latency.
constexpr int kSpreadThreads = 512;
constexpr int kSpreadItems = 8;
constexpr int kSpreadTile = kSpreadThreads * kSpreadItems;  // keys per CTA

__global__ void __launch_bounds__(kSpreadThreads) k_sort_count(const uint32_t* __restrict__ keys, int64_t n, int shift,
                                                               int nd, SortState* st) {
  chain_wait();
  extern __shared__ __align__(16) uint32_t sbuf[];
  __shared__ uint32_t s_w[kSpreadThreads / 32];
  __shared__ bool last;
  uint32_t* const cnt = sbuf;  // [nd]
  const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int d = t; d < nd; d += kSpreadThreads) cnt[d] = 0u;
  const int64_t base = int64_t(blockIdx.x) * kSpreadTile;
  uint32_t k[kSpreadItems];
#pragma unroll
  for (int i = 0; i < kSpreadItems; ++i) {
    const int64_t o = base + i * kSpreadThreads + int64_t(t);
    k[i] = o < n ? keys[o] : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSpreadItems; ++i) {
    const bool ok = base + i * kSpreadThreads + int64_t(t) < n;
    const unsigned d = k[i] >> shift, d0 = __shfl_sync(0xffffffffu, d, 0);
    if (__all_sync(0xffffffffu, ok && d == d0)) {  // 32 keys of one digit (nearly sorted input): one atomic
      if (lane == 0) atomicAdd(&cnt[d0], 32u);
    } else if (ok) {
      atomicAdd(&cnt[d], 1u);
    }
  }
  __syncthreads();
  for (int d = t; d < nd; d += kSpreadThreads)
    if (cnt[d]) atomicAdd(&st->tot[d], cnt[d]);
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // starts of the buckets: exclusive scan of the totals, which go back to zero
  const int per = (nd + kSpreadThreads - 1) / kSpreadThreads;
  uint32_t sum = 0;
  for (int i = 0; i < per; ++i) {
    const int d = per * int(t) + i;
    if (d < nd) {
      const uint32_t c = __ldcg(&st->tot[d]);
      cnt[d] = c;
      st->tot[d] = 0u;
      sum += c;
    }
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= unsigned(o)) inc += x;
  }
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  uint32_t off = inc - sum;
  for (unsigned w = 0; w < warp; ++w) off += s_w[w];
  for (int i = 0; i < per; ++i) {
    const int d = per * int(t) + i;
    if (d < nd) {
      st->cur[d] = off;
      off += cnt[d];
    }
  }
  if (t == 0) st->ticket = 0u;
}

__global__ void __launch_bounds__(kSpreadThreads) k_sort_spread(const uint32_t* __restrict__ keys, int64_t n, int shift,
                                                                int nd, SortState* st, uint32_t* __restrict__ kout,
                                                                uint32_t* __restrict__ vout, int* err) {
  chain_wait();
  extern __shared__ __align__(16) uint32_t sbuf[];
  uint32_t* const cnt = sbuf;  // [nd]: counts, then the place of the CTA's first key of the digit
  const unsigned t = threadIdx.x, lane = t & 31;
  for (int d = t; d < nd; d += kSpreadThreads) cnt[d] = 0u;
  const int64_t base = int64_t(blockIdx.x) * kSpreadTile;
  uint32_t k[kSpreadItems], r[kSpreadItems];
#pragma unroll
  for (int i = 0; i < kSpreadItems; ++i) {
    const int64_t o = base + i * kSpreadThreads + int64_t(t);
    k[i] = o < n ? keys[o] : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSpreadItems; ++i) {
    const bool ok = base + i * kSpreadThreads + int64_t(t) < n;
    const unsigned d = k[i] >> shift, d0 = __shfl_sync(0xffffffffu, d, 0);
    r[i] = 0u;
    if (__all_sync(0xffffffffu, ok && d == d0)) {
      if (lane == 0) r[i] = atomicAdd(&cnt[d0], 32u);
      r[i] = __shfl_sync(0xffffffffu, r[i], 0) + lane;
    } else if (ok) {
      r[i] = atomicAdd(&cnt[d], 1u);
    }
  }
  __syncthreads();
  for (int d = t; d < nd; d += kSpreadThreads) {
    const uint32_t c = cnt[d];
    if (c) cnt[d] = atomicAdd(&st->cur[d], c);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSpreadItems; ++i) {
    const int64_t o = base + i * kSpreadThreads + int64_t(t);
    if (o < n) {
      const uint32_t p = cnt[k[i] >> shift] + r[i];
      if (p < n) {
        kout[p] = k[i];
        vout[p] = uint32_t(o);
      } else {
        atomicOr(err, kErrSort);
      }
    }
  }
}

// Radius order of the state as component arrays: sorted position j takes the record src[v]
// (one particle: whole sectors), which the moments and field kernels read.
template <class T> struct SoA { T* d[6]; uint32_t* id; };
template <class T> __device__ __forceinline__ void put_part(const SoA<T>& dst, int64_t j, const Part<T>& p) {
  dst.d[0][j] = p.x; dst.d[1][j] = p.y; dst.d[2][j] = p.z;
  dst.d[3][j] = p.vx; dst.d[4][j] = p.vy; dst.d[5][j] = p.vz;
  dst.id[j] = p.id;
}

// Sort of one bucket (with st; or of the whole array k1 without) in one CTA, and the gather of
// its particles into radius order. The keys of a bucket spread over its range like the density
// over r^2, so a second digit of sb bits with about one key per value leaves almost nothing to
// sort: the CTA counts the digits (shared atomics), scans the counts, places (key, slot) by
// digit in any order, and each placed key finds its rank among the few of its digit by comparing
// (key, slot): the order of a stable sort of the input slots by key, whatever the order of the
// atomics. A bucket of more than cap keys is placed by digit in global memory and ranked in ranges
// of digits that fit: its work grows with its keys. A comparison costs some 0.08 ns of the CTA's
// time, a byte pass of eight ballots 1 ns per key: beyond kBsMeanRun keys in a key's digit on average
// (or kBsMaxRun in one: one thread's share) the bucket goes through stable byte passes in L2
// instead. Sort and gather of uneven sets (us; rounds that each read the whole bucket and a line
// at kBsMaxRun alone -> this; byte passes by slot and by key for every bucket): N = 3e5 with nine
// tenths of the particles in 0.03 of the range of r^2 351 -> 232 (569), in 0.01 2037 -> 955 (1611), in
// 0.003 8104 -> 1756 (3001); N = 2e6 with 0.03 445 -> 362 (563), 0.01 2585 -> 1234 (1488), 0.001 13770
// -> 8120 (13860); 30 discrete radii 1488 -> 1096 (1472). One CTA still takes all of a bucket.
// k1 (v1): keys and input slots of the buckets (without st the keys in input order, v1 scratch);
// k0, v0: scratch for the byte passes. tb: leading key bits the same in all of a bucket;
// sb <= 32 - tb, 2^sb >= NT.
// Bound by the latency of the shared atomics, of the loads from L2 and of the gather: three CTAs
// of 512 threads per SM keep more of them in flight than two with more registers (N = 2e6: a step
// of 0.759 ms against 0.764; N = 7e5 0.231 and 0.234). A bucket's three byte passes of eight
// ballots per 32 keys took 0.067 ms of the 0.111 ms sort of 2e6 keys and the gather a kernel of
// 0.024 ms; this kernel 0.040 with the gather, sort and gather 0.138 -> 0.069. N = 3001 0.032 ->
// 0.012, N = 20000 0.027 -> 0.0175, N = 5e5 0.051 -> 0.027.
constexpr int kBsMaxRun = 256, kBsMeanRun = 32;
constexpr int kBsTies = 32;  // ties of one key ordered by counting; more by three passes over the slots
constexpr size_t kBsRankBytes = 8;  // shared memory per key: key and slot
constexpr int kBsThreads = 512, kBsPerSM = 3;  // CTA of a bucket, resident per SM
constexpr int kBsOneThreads = 1024;  // the one CTA of a small array
static_assert(kBsThreads >= 256 && kBsOneThreads >= 256, "256 threads scan the byte counts");

// Stable byte passes over the bucket start .. start + len by the key bits in which its keys differ, and
// the gather. The whole array (in_slots) is in the order of its slots already. In a bucket ties are then
// ordered by counting the slots among them, or by passes over the slots (the bytes that n_all has) before
// those over the keys: at once where more than kBsTies keys share a value on average, afterwards where a
// run of ties is longer. A function of its own: inlined, it makes the kernel spill for all its buckets
// (52 bytes with 512 threads, so none; sort of N = 1e5: 20.5 us, so 19.8; 2e6: 73.0 and 71.5).
template <class T, int NT>
__device__ __noinline__ void bucket_bytes(uint32_t* k1, uint32_t* v1, uint32_t* k0, uint32_t* v0, int64_t start, int64_t len,
                                          int64_t n_all, bool in_slots, const Part<T>* src, const SoA<T>& dst, int* err) {
  extern __shared__ __align__(16) uint32_t sbuf[];
  __shared__ uint32_t s_diff;
  const unsigned t = threadIdx.x, lane = t & 31;
  BsShared<NT>& sh = *reinterpret_cast<BsShared<NT>*>(sbuf);
  uint32_t *ak = k1, *av = v1, *dk = k0, *dv = v0;
  if (t == 0) s_diff = 0u;
  uint32_t diff = 0;
  {
    const uint32_t first = ak[0];
#pragma unroll 4
    for (int64_t i = t; i < len; i += NT) diff |= ak[i] ^ first;
  }
  if (in_slots)
    for (int64_t i = t; i < len; i += NT) av[i] = uint32_t(i);
  __syncthreads();
  diff = __reduce_or_sync(0xffffffffu, diff);
  if (lane == 0) atomicOr(&s_diff, diff);
  __syncthreads();
  diff = s_diff;
  auto pass = [&](bool by_slot, int shift) {
    if (t < 256) sh.cnt[t] = 0u;
    __syncthreads();
    count_byte<NT>(by_slot ? av : ak, len, shift, sh.cnt);
    __syncthreads();
    if (by_slot) bucket_pass<NT>(av, ak, dv, dk, int(len), shift, sh);
    else bucket_pass<NT>(ak, av, dk, dv, int(len), shift, sh);
    uint32_t* x = ak; ak = dk; dk = x;
    x = av; av = dv; dv = x;
  };
  auto by_slot = [&]() {
    for (int shift = 0; shift < 32 && ((n_all - 1) >> shift) != 0; shift += 8) pass(true, shift);
  };
  auto by_key = [&]() {
    for (int shift = 0; shift < 32; shift += 8)
      if ((diff >> shift) & 255u) pass(false, shift);
  };
  bool in_order = in_slots || int64_t(diff) * kBsTies < len;  // ties come out in the order of their slots
  if (!in_slots && in_order) by_slot();
  by_key();
  if (!in_order) {
    bool ties = false;
    for (int64_t i = t; i + kBsTies < len; i += NT) ties = ties || ak[i] == ak[i + kBsTies];
    if (__syncthreads_or(ties)) {
      by_slot();
      by_key();
      in_order = true;
    }
  }
  constexpr int G = 4;  // gathers in flight per thread
  const int m = int(len);
  for (int i0 = 0; i0 < m; i0 += NT * G) {
    int at[G];
    uint32_t from[G];
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const int i = at[u] = i0 + u * NT + int(t);
      from[u] = 0u;
      if (i >= m) continue;
      const uint32_t key = ak[i], v = av[i];
      for (int q = i - 1; !in_order && q >= 0 && ak[q] == key; --q) at[u] -= av[q] > v;
      for (int q = i + 1; !in_order && q < m && ak[q] == key; ++q) at[u] += av[q] < v;
      from[u] = v < n_all ? v : 0u;
      if (v >= n_all) atomicOr(err, kErrSort);
    }
    Part<T> x[G];
#pragma unroll
    for (int u = 0; u < G; ++u) x[u] = src[from[u]];
#pragma unroll
    for (int u = 0; u < G; ++u)
      if (i0 + u * NT + int(t) < m) put_part<T>(dst, start + at[u], x[u]);
  }
}

template <class T, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_bucket_sort(uint32_t* k1, uint32_t* v1, uint32_t* k0, uint32_t* v0,
                                                          const SortState* __restrict__ st, int64_t n_all, int cap,
                                                          int tb, int sb, const Part<T>* __restrict__ src,
                                                          const __grid_constant__ SoA<T> dst, int* err) {
  chain_wait();
  extern __shared__ __align__(16) uint32_t sbuf[];
  __shared__ uint32_t s_w[NT / 32];
  const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t* const cnt = sbuf;                // [2^sb + 1]
  uint32_t* const ks = cnt + (1 << sb) + 1;  // [cap]
  uint32_t* const vs = ks + cap;             // [cap]
  int64_t start = 0, len = n_all;
  if (st) {  // the cursors are the buckets' ends now
    start = blockIdx.x ? st->cur[blockIdx.x - 1] : 0u;
    len = int64_t(st->cur[blockIdx.x]) - start;
    if (len < 0 || start + len > n_all) {  // never with a sort state in order; uniform over the CTA
      if (t == 0) atomicOr(err, kErrSort);
      return;
    }
  }
  if (len == 0) return;  // uniform over the CTA
  const auto slot = [&](uint32_t v) {  // a slot that the spread did not write is no particle
    if (v < n_all) return v;
    atomicOr(err, kErrSort);
    return 0u;
  };
  const uint32_t* const sk = k1 + start;
  const uint32_t* const sv = v1 + start;
  {
    const int n = int(len), shift = 32 - sb;
    constexpr int U = 4;  // keys per thread in flight
    const bool once = n <= NT * U;  // each thread's keys, slots and places in their digits stay in registers
    uint32_t k[U], v[U], r[U];
    for (int d = t; d <= 1 << sb; d += NT) cnt[d] = 0u;
    auto load = [&](int i0) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * NT + int(t);
        k[u] = i < n ? sk[i] : 0u;
        v[u] = st ? (i < n ? sv[i] : 0u) : unsigned(i);
      }
    };
    auto count = [&](int i0) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        r[u] = i0 + u * NT + int(t) < n ? atomicAdd(&cnt[((k[u] << tb) >> shift) + 1], 1u) : 0u;
    };
    if (once) load(0);
    __syncthreads();
    if (once) {
      count(0);
    } else {
      for (int i0 = 0; i0 < n; i0 += NT * U) {
        load(i0);
        count(i0);
      }
    }
    __syncthreads();
    // scan of the counts, each thread 2^sb / NT of them: to the digits' ends (cnt[s + 1], so
    // cnt[s] is the start of s), or to their starts, which become cursors and so the ends
    const int per = (1 << sb) / NT;
    uint32_t* const mine = cnt + per * t + 1;
    uint32_t sum = 0, big = 0;
    for (int d = 0; d < per; ++d) {
      const uint32_t c = mine[d];
      sum += c;
      big = c > big ? c : big;
    }
    bool rank = true;
    if (__syncthreads_or(big > unsigned(kBsMeanRun))) {  // a crowded digit: what the comparisons would be
      if (t == 0) s_w[0] = 0u;
      rank = !__syncthreads_or(big > unsigned(kBsMaxRun));
      if (rank) {
        uint32_t pairs = 0;
        for (int d = 0; d < per; ++d) pairs += mine[d] * mine[d];
        atomicAdd(s_w, pairs);
        __syncthreads();
        rank = s_w[0] <= uint32_t(kBsMeanRun) * uint32_t(n);
        __syncthreads();
      }
    }
    if (rank) {
      uint32_t inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= unsigned(o)) inc += x;
      }
      if (lane == 31) s_w[warp] = inc;
      __syncthreads();
      uint32_t off = inc - sum;
      for (unsigned w = 0; w < warp; ++w) off += s_w[w];
      for (int d = 0; d < per; ++d) {
        const uint32_t end = off + mine[d];
        mine[d] = once ? end : off;
        off = end;
      }
      __syncthreads();
      // One range of digits for all of a bucket, but for an overfull one: that is placed in global
      // memory (k0, v0) and comes back in ranges [d0, d1) of at most cap keys each.
      const uint32_t digits = 1u << sb;
      const bool over = n > cap;
      auto place = [&](int i0, uint32_t* kd, uint32_t* vd) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t s = (k[u] << tb) >> shift;
          if (i0 + u * NT + int(t) < n) {
            const uint32_t p = once ? cnt[s] + r[u] : atomicAdd(&cnt[s + 1], 1u);
            kd[p] = k[u];
            vd[p] = v[u];
          }
        }
      };
      if (once) {
        place(0, ks, vs);
      } else {
        for (int i0 = 0; i0 < n; i0 += NT * U) {
          load(i0);
          place(i0, over ? k0 + start : ks, over ? v0 + start : vs);
        }
      }
      __syncthreads();  // the cursors stand at the digits' ends: cnt[s] is the start of s
      for (uint32_t d0 = 0; d0 < digits;) {
        uint32_t base = 0, d1 = digits, m = n;
        if (over) {
          base = cnt[d0];
          uint32_t lo = d0 + 1, hi = digits;  // the last d1 with start(d1) - base <= cap
          while (lo < hi) {
            const uint32_t mid = (lo + hi + 1) / 2;
            if (cnt[mid] - base <= uint32_t(cap)) lo = mid;
            else hi = mid - 1;
          }
          d1 = lo;
          m = cnt[d1] - base;
          for (uint32_t i = t; i < m; i += NT) {
            ks[i] = k0[start + base + i];
            vs[i] = v0[start + base + i];
          }
          __syncthreads();
        }
        constexpr int G = MINB == 1 ? 4 : 2;  // gathers in flight per thread
        for (uint32_t p0 = 0; p0 < m; p0 += NT * G) {
          uint32_t at[G], from[G];
#pragma unroll
          for (int u = 0; u < G; ++u) {
            const uint32_t p = p0 + u * NT + t;
            at[u] = from[u] = 0u;
            if (p >= m) continue;
            const uint32_t key = ks[p], s = (key << tb) >> shift, b = cnt[s] - base, e = cnt[s + 1] - base;
            from[u] = vs[p];
            at[u] = b;
#pragma unroll 1  // a digit has few keys (sort of N = 5e5: 33.6 us, unrolled 34.2; 2e6: 71.1 and 71.5)
            for (uint32_t q = b; q < e; ++q) {
              const uint32_t kq = ks[q];
              at[u] += kq < key || (kq == key && vs[q] < from[u]) ? 1u : 0u;
            }
            from[u] = slot(from[u]);
          }
          Part<T> x[G];
#pragma unroll
          for (int u = 0; u < G; ++u) x[u] = src[from[u]];
#pragma unroll
          for (int u = 0; u < G; ++u)
            if (p0 + u * NT + t < m) put_part<T>(dst, start + base + at[u], x[u]);
        }
        d0 = d1;
        if (d0 < digits) __syncthreads();  // the placed keys have been read
      }
      return;
    }
  }
  __syncthreads();  // the counts have been read
  bucket_bytes<T, NT>(k1 + start, v1 + start, k0 + start, v0 + start, start, len, n_all, !st, src, dst, err);
}

// Largest N for the bucket sort (2930 keys a bucket on average); larger arrays take the four global
// passes. kSortDigits: with 4096 digits, 3906 keys a bucket at N = 1.6e7, each bucket's keys are
// read twice; 8192 leave one round of loads for most: sort and gather 0.670 -> 0.434 ms, a step
// 10.96 -> 10.73.
constexpr int64_t kBucketSortMaxN = 24000000;
constexpr int kBsCapMax = 13312;
constexpr int kBsBitsMax = 13;
// up to here one CTA sorts everything (0.011 ms; at 6000 keys 0.0145 against 0.015)
constexpr int64_t kBsSingleN = 4096;
// Digits of the first pass. Alone on the GPU 256 buckets (the most parallel) up to kBsSmallN keys
// (N = 3e5: a step of 0.0892 ms, with 512 0.0904; 5e5: 0.0757 and 0.0761), beyond as many as
// leave at most kBsMean keys on average, so that one round of loads holds a bucket (N = 2e6: 0.774
// ms a step with up to 2048, 0.761 with 1024, 0.778 with 512). Sharing it (a batch), fewer and
// fuller CTAs.
constexpr int64_t kBsSmallN = 1 << 19, kBsMean = 1024;
inline int sort_digit_bits(int64_t n, bool shared_gpu) {
  int b = shared_gpu ? 1 : 8;
  const int64_t mean = n > kBsSmallN ? kBsMean : 2 * kBsMean;
  while ((n >> b) > mean && (1 << b) < kSortDigits) ++b;
  return b;
}
int sort_digits(int64_t n) { return 1 << sort_digit_bits(n, false); }
// Shared-memory capacity for buckets of `mean` keys on average (a larger one takes several ranges)
inline int bucket_cap(int64_t mean) {
  int64_t c = (mean + mean / 4 * 3 + 255) / 256 * 256;
  if (c < 2048) c = 2048;
  return int(c < kBsCapMax ? c : kBsCapMax);
}
// Bits of the second digit for segments of `mean` keys: about one key per value
inline int bucket_bits(int64_t mean, int threads) {
  int sb = 0;
  while ((1 << sb) < threads || ((int64_t(1) << sb) < mean && sb < kBsBitsMax)) ++sb;
  return sb;
}
template <int NT> inline size_t bucket_smem(int cap, int sb) {
  const size_t rank = (size_t(4) << sb) + 4 + kBsRankBytes * size_t(cap), pass = sizeof(BsShared<NT>);
  return rank > pass ? rank : pass;
}

cudaError_t set_sort_attributes() {
  const int most = int(bucket_smem<kBsOneThreads>(kBsCapMax, kBsBitsMax));
  cudaError_t e = cudaFuncSetAttribute(k_bucket_sort<float, kBsOneThreads, 1>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_bucket_sort<double, kBsOneThreads, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             most);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_bucket_sort<float, kBsThreads, kBsPerSM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             most);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_bucket_sort<double, kBsThreads, kBsPerSM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             most);
  return e;
}

template <class T>
const uint32_t* launch_radix_sort(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, void* scratch, int64_t n,
                                  int first_byte, const Part<T>* src, T* const* dst, uint32_t* id_dst, int* err,
                                  LaunchSeq& seq, bool shared_gpu) {
  if (n <= 1) return v0;
  SoA<T> d;
  for (int c = 0; c < 6; ++c) d.d[c] = dst[c];
  d.id = id_dst;
  SortState* const st = static_cast<SortState*>(scratch);
  if (first_byte == 0 && n <= kBsSingleN) {
    const int cap = int((n + 255) / 256 * 256), sb = bucket_bits(n, kBsOneThreads);
    seq(k_bucket_sort<T, kBsOneThreads, 1>, 1, kBsOneThreads, bucket_smem<kBsOneThreads>(cap, sb), k0, v0, k1, v1,
        nullptr, n, cap, 0, sb, src, d, err);
    return nullptr;
  }
  if (first_byte == 0 && n <= kBucketSortMaxN) {
    const int tb = sort_digit_bits(n, shared_gpu), nd = 1 << tb, shift = 32 - tb;
    const int64_t mean = n >> tb;
    const int cap = bucket_cap(mean), sb = bucket_bits(mean, kBsThreads);
    const unsigned blocks = unsigned((n + kSpreadTile - 1) / kSpreadTile);
    seq(k_sort_count, blocks, kSpreadThreads, sizeof(uint32_t) * nd, k0, n, shift, nd, st);
    seq(k_sort_spread, blocks, kSpreadThreads, sizeof(uint32_t) * nd, k0, n, shift, nd, st, k1, v1, err);
    seq(k_bucket_sort<T, kBsThreads, kBsPerSM>, unsigned(nd), kBsThreads, bucket_smem<kBsThreads>(cap, sb), k1, v1, k0,
        v0, st, n, cap, tb, sb, src, d, err);
    return nullptr;
  }
  const int64_t nblk = sort_blocks(n);
  uint32_t* hist = reinterpret_cast<uint32_t*>(st + 1);
  uint32_t* rowtot = hist + 256 * nblk;
  uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
  for (int pass = first_byte; pass < 4; ++pass) {
    const int shift = 8 * pass;
    seq(k_sort_hist, unsigned(nblk), kSortThreads, 0, ki, n, shift, nblk, hist);
    seq(k_sort_rowscan, 256, kSortThreads, 0, hist, nblk, rowtot);
    seq(k_sort_scatter, unsigned(nblk), kSortThreads, 0, ki, vi, ko, vo, n, shift, nblk, hist, rowtot);
    uint32_t* tk = ki; ki = ko; ko = tk;
    uint32_t* tv = vi; vi = vo; vo = tv;
  }
  return vi;
}

// ============================================================================
// State movement
// ============================================================================
// Gather of the state into radius order by a permutation (very large arrays; the bucket
// sort gathers itself).
template <class T>
__global__ void k_reorder(const Part<T>* __restrict__ src, SoA<T> dst, const uint32_t* __restrict__ perm,
                          int64_t n) {
  chain_wait();
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  put_part<T>(dst, j, src[perm[j]]);
}

template <class T>
void launch_reorder(const Part<T>* src, T* const* dst, uint32_t* id_dst, const uint32_t* perm, int64_t n,
                    LaunchSeq& seq) {
  SoA<T> d;
  for (int c = 0; c < 6; ++c) d.d[c] = dst[c];
  d.id = id_dst;
  seq(k_reorder<T>, unsigned((n + 255) / 256), 256, 0, src, d, perm, n);
}

// Radius keys of the state in its storage order (after a load or a field
// evaluation; a step's field kernel writes the next keys itself).
template <class T>
__global__ void k_keys(const Part<T>* __restrict__ st, uint32_t* __restrict__ key, uint32_t* __restrict__ kidx,
                       int64_t n, RadiusKey rk) {
  chain_wait();
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const Part<T> p = st[j];
  key[j] = radius_key<T>(p.x, p.y, p.z, rk);
  kidx[j] = uint32_t(j);
}

template <class T>
void launch_keys(const Part<T>* st, uint32_t* key, uint32_t* kidx, int64_t n, double r_out, LaunchSeq& seq) {
  seq(k_keys<T>, unsigned((n + 255) / 256), 256, 0, st, key, kidx, n, make_radius_key(r_out));
}

// FP64 -> FP32 rounding to nearest, ties to even (IEEE 754 binary64 ->
// binary32), in integer operations: FP64 arithmetic, conversions included,
// runs at a small fraction of the FP32 rate on this part and bound the load
// kernel. Normal results keep the top 23 of the 52 mantissa bits and round on
// the other 29 (a carry steps the exponent, up to infinity at the top of the
// range); subnormal results shift the full 53-bit significand into the
// subnormal units and round on the shifted-out bits; overflow gives infinity,
// NaN stays a (quiet) NaN.
__device__ __forceinline__ float f64_to_f32_rn(double d) {
  const uint64_t b = uint64_t(__double_as_longlong(d));
  const uint32_t sign = uint32_t(b >> 32) & 0x80000000u;
  const int e = int(b >> 52) & 0x7ff;
  const uint64_t m = b & 0xfffffffffffffull;
  uint32_t bits;
  if (e >= 897 && e <= 1150) {  // normal FP32 result
    const uint32_t top = uint32_t(m >> 29), rest = uint32_t(m) & 0x1fffffffu;
    bits = (uint32_t(e - 896) << 23) | top;
    if (rest > 0x10000000u || (rest == 0x10000000u && (top & 1u))) bits += 1u;
  } else if (e == 0x7ff) {  // infinity, NaN
    bits = 0x7f800000u | (m ? (0x400000u | uint32_t(m >> 29)) : 0u);
  } else if (e > 1150) {    // overflow
    bits = 0x7f800000u;
  } else if (e >= 873) {    // subnormal result: M 2^(e - 926) units of 2^-149
    const uint64_t M = m | (1ull << 52);
    const int sh = 926 - e;  // 30 .. 53
    const uint64_t q = M >> sh, r = M & ((1ull << sh) - 1), h = 1ull << (sh - 1);
    bits = uint32_t(q) + ((r > h || (r == h && (q & 1u))) ? 1u : 0u);
  } else {                  // below half the smallest subnormal
    bits = 0u;
  }
  return __uint_as_float(sign | bits);
}
// FP32 -> FP64, exact, in integer operations: the exponent rebiased and the
// mantissa widened; a subnormal is normalised from its leading bit.
__device__ __forceinline__ double f32_to_f64(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint64_t sign = uint64_t(u & 0x80000000u) << 32;
  const uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  uint64_t bits;
  if (e == 255u) {
    bits = 0x7ff0000000000000ull | (uint64_t(m) << 29);
  } else if (e != 0u) {
    bits = (uint64_t(e + 896u) << 52) | (uint64_t(m) << 29);
  } else if (m == 0u) {
    bits = 0;
  } else {  // m 2^-149, leading bit at p
    const int p = 31 - __clz(m);
    bits = (uint64_t(p - 149 + 1023) << 52) | ((uint64_t(m) << (52 - p)) & 0xfffffffffffffull);
  }
  return __longlong_as_double(int64_t(sign | bits));
}
template <class T> __device__ __forceinline__ T narrow(double d);
template <> __device__ __forceinline__ float narrow<float>(double d) { return f64_to_f32_rn(d); }
template <> __device__ __forceinline__ double narrow<double>(double d) { return d; }
template <class T> __device__ __forceinline__ double widen(T v);
template <> __device__ __forceinline__ double widen<float>(float v) { return f32_to_f64(v); }
template <> __device__ __forceinline__ double widen<double>(double v) { return v; }

// Host FP64 [n][3] positions and velocities into the state, ids 0..n-1, with
// the radius keys of that order, so that the first step after a load needs no
// separate key pass.
template <class T>
__global__ void k_load(const double* __restrict__ xs, const double* __restrict__ vs,
                       const uint32_t* __restrict__ ids, Part<T>* __restrict__ st, uint32_t* __restrict__ key,
                       uint32_t* __restrict__ kidx, int64_t n, double r_out2, RadiusKey rk, int* err) {
  const int64_t j0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t j = j0 < n ? j0 : n - 1;  // (every thread votes below)
  double v[6];
  bool fin = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    v[c] = xs[3 * j + c];
    v[3 + c] = vs[3 * j + c];
  }
  // finiteness from the exponent bits (integer work: FP64 operations run at a
  // small fraction of the FP32 rate on this part and bound this kernel)
#pragma unroll
  for (int c = 0; c < 6; ++c)
    fin = fin && ((uint32_t(__double_as_longlong(v[c]) >> 32) & 0x7ff00000u) != 0x7ff00000u);
  Part<T> p;
  p.x = narrow<T>(v[0]); p.y = narrow<T>(v[1]); p.z = narrow<T>(v[2]);
  p.vx = narrow<T>(v[3]); p.vy = narrow<T>(v[4]); p.vz = narrow<T>(v[5]);
  p.id = ids ? ids[j] : uint32_t(j);
  // range test and radius key (radius_key's two forms, with r^2 shared)
  bool inside;
  uint32_t k;
  bool fx = false;
  if constexpr (sizeof(T) == 4) fx = key_fx_applies(p.x, p.y, p.z, rk);
  if (fx) {
    const uint64_t R2 = r2_fx(float(p.x), float(p.y), float(p.z));
    inside = R2 > kFxOne && R2 < rk.rout2_fx;
    k = key_of_fx(R2, rk);
  } else {
    const double xd = widen<T>(p.x), yd = widen<T>(p.y), zd = widen<T>(p.z);
    const double r2 = xd * xd + yd * yd + zd * zd;
    inside = r2 > 1.0 && r2 < r_out2;
    k = key_of_r2(r2, rk);
  }
  // one atomic per CTA: the flags stand in host memory, where atomics are done one after the other
  // (8e6 bad particles with one per warp 4.9 ms, a good load 2.2)
  const bool nan = __syncthreads_or(!fin), out = __syncthreads_or(fin && !inside);
  if (threadIdx.x == 0 && (nan || out)) atomicOr(err, (nan ? kErrNaN : 0) | (out ? kErrRange : 0));
  if (j0 >= n) return;
  st[j] = p;
  key[j] = k;
  kidx[j] = uint32_t(j);
}

template <class T>
void launch_load(const double* x, const double* v, const uint32_t* ids, Part<T>* st, uint32_t* key,
                 uint32_t* kidx, int64_t n, double r_out, int* err, cudaStream_t s) {
  k_load<T><<<unsigned((n + 255) / 256), 256, 0, s>>>(x, v, ids, st, key, kidx, n, r_out * r_out,
                                                      make_radius_key(r_out), err);
}

template <class T>
__global__ void k_state_dump(const Part<T>* __restrict__ st, double* __restrict__ x, double* __restrict__ v,
                             uint32_t* __restrict__ id, int64_t n) {
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const Part<T> p = st[j];
  x[3 * j] = p.x; x[3 * j + 1] = p.y; x[3 * j + 2] = p.z;
  v[3 * j] = p.vx; v[3 * j + 1] = p.vy; v[3 * j + 2] = p.vz;
  id[j] = p.id;
}

template <class T>
void launch_state_dump(const Part<T>* st, double* x, double* v, uint32_t* id, int64_t n, cudaStream_t s) {
  k_state_dump<T><<<unsigned((n + 255) / 256), 256, 0, s>>>(st, x, v, id, n);
}

// out[id[j]][c] = comp_c[j] for c < nc (field values in radius order to id order)
template <class T> struct Ptr6 { const T* d[6]; };
template <class T>
__global__ void k_scatter_by_id(Ptr6<T> p, int nc, const uint32_t* __restrict__ id,
                                double* __restrict__ out, int64_t n) {
  chain_wait();
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int64_t k = id[j];
  if (k >= n) return;  // only after a sort that ended with kErrSort
  for (int c = 0; c < nc; ++c) out[k * nc + c] = double(p.d[c][j]);
}

template <class T>
void launch_scatter_by_id(const T* const* comps, int ncomp, const uint32_t* id, double* out, int64_t n,
                          LaunchSeq& seq) {
  Ptr6<T> p;
  for (int c = 0; c < ncomp; ++c) p.d[c] = comps[c];
  seq(k_scatter_by_id<T>, unsigned((n + 255) / 256), 256, 0, p, ncomp, id, out, n);
}

// The state in id order: x[id][3] and v[id][3], FP64. Up to kGatherMinN particles
// each record is scattered to its id's place; beyond, where the outputs (48 bytes
// per particle) leave L2 and every scattered 24-byte piece costs two sectors read and
// written, the inverse order is written first (4 bytes per particle) and each id's
// record gathered, one sector, so that the outputs are written in order: N = 1.6e7:
// 1.94 -> 0.60 ms, N = 2e6: 0.147 -> 0.065, N = 5e5: 0.028 -> 0.021 (N = 3e5: 0.014
// against 0.016).
constexpr int64_t kGatherMinN = 393216;
template <class T>
__global__ void k_state_out(const Part<T>* __restrict__ st, double* __restrict__ x, double* __restrict__ v,
                            int64_t n) {
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const Part<T> p = st[j];
  const int64_t k = p.id;
  if (k >= n) return;  // only after a sort that ended with kErrSort; so below
  x[3 * k] = p.x; x[3 * k + 1] = p.y; x[3 * k + 2] = p.z;
  v[3 * k] = p.vx; v[3 * k + 1] = p.vy; v[3 * k + 2] = p.vz;
}
template <class T>
__global__ void k_inverse_ids(const Part<T>* __restrict__ st, uint32_t* __restrict__ inv, int64_t n) {
  const int64_t j = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (j < n && st[j].id < n) inv[st[j].id] = uint32_t(j);
}
template <class T>
__global__ void k_state_gather(const Part<T>* __restrict__ st, const uint32_t* __restrict__ inv,
                               double* __restrict__ x, double* __restrict__ v, int64_t n) {
  chain_wait();
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int64_t j = inv[k];
  if (j >= n) return;
  const Part<T> p = st[j];
  x[3 * k] = p.x; x[3 * k + 1] = p.y; x[3 * k + 2] = p.z;
  v[3 * k] = p.vx; v[3 * k + 1] = p.vy; v[3 * k + 2] = p.vz;
}

template <class T>
void launch_state_out(const Part<T>* st, double* x, double* v, uint32_t* inv, int64_t n, cudaStream_t s) {
  LaunchSeq seq(s);
  const unsigned blocks = unsigned((n + 255) / 256);
  if (n < kGatherMinN) {
    seq(k_state_out<T>, blocks, 256, 0, st, x, v, n);
  } else {
    seq(k_inverse_ids<T>, blocks, 256, 0, st, inv, n);
    seq(k_state_gather<T>, blocks, 256, 0, st, static_cast<const uint32_t*>(inv), x, v, n);
  }
}

// ============================================================================
// Scans of the tile moments (FP64 accumulation)
// ============================================================================
// Tile scan: the in-group scans of the tile sums agg[u][tile] over the tw
// tiles of whole groups (row stride ts). One warp task = 128 consecutive tiles of
// one row = 4 groups; lane l holds tiles 4l..4l+3 (one vector load), so a
// group is 8 lanes. Each lane sums its 4 tiles in order, an 8-lane shuffle
// scan gives the lane's offset, and the lane writes its 4 results with one
// vector store. Rs rows (u even): exclusive prefix towards higher tiles; Is
// rows (u odd): exclusive suffix towards lower tiles; each summed in its own
// direction (no total minus a partial sum, which would cancel). The group
// total (the inclusive sum at the far end) goes to gagg[g][u] in FP64. Each
// warp takes kTsTasks consecutive tasks and issues their loads first.
// ============================================================================

// Compensated partial sums of the in-group scans. In FP32 every partial sum is
// the unevaluated pair hi + lo: hi is the plain running sum and lo collects the
// rounding error of every addition, which Knuth's TwoSum gives exactly, so a
// sum over the 1024 particles of a scan group keeps about twice the working
// precision (the radius-ordered scans are where cancellation sets the
// accuracy). The results are rounded to FP32 once (hi + lo), the group totals
// to FP64. In FP64 the sums are plain.
template <class T> struct CSum { T hi, lo; };
template <class T> __device__ __forceinline__ CSum<T> cs_add(CSum<T> a, CSum<T> b) {
  if constexpr (sizeof(T) == 4) {
    const T s = a.hi + b.hi;
    const T bb = s - a.hi;
    const T e = (a.hi - (s - bb)) + (b.hi - bb);  // a.hi + b.hi = s + e exactly
    return {s, (a.lo + b.lo) + e};
  } else {
    return {a.hi + b.hi, T(0)};
  }
}
template <class T> __device__ __forceinline__ T cs_round(CSum<T> v) { return v.hi + v.lo; }
template <class T> __device__ __forceinline__ CSum<T> cs_of(T v) { return {v, T(0)}; }
template <class T> __device__ __forceinline__ CSum<T> cs_shfl_down(CSum<T> v, int d) {
  return {__shfl_down_sync(0xffffffffu, v.hi, d, 8), __shfl_down_sync(0xffffffffu, v.lo, d, 8)};
}
template <class T> __device__ __forceinline__ CSum<T> cs_shfl_up(CSum<T> v, int d) {
  return {__shfl_up_sync(0xffffffffu, v.hi, d, 8), __shfl_up_sync(0xffffffffu, v.lo, d, 8)};
}
template <class T> __device__ __forceinline__ double cs_double(CSum<T> v) { return double(v.hi) + double(v.lo); }

// In-group scans of the tile sums. A CTA takes 32 rows (components u) x 128
// tiles (4 scan groups) of agg[u][tile]: each warp scans 4 rows, one V4 of 4
// tiles per lane (a 4-element in-lane scan plus an 8-lane shuffle scan per
// group), and the CTA writes the results transposed, pfx[tile][u], through
// shared memory, so that the field kernel reads the carries of one tile as
// contiguous lines. Is rows (u odd) get exclusive suffixes, Rs rows (u even)
// exclusive prefixes; the group totals go to gagg[g][u] in FP64, converted by full
// warps after the scans (by the four lanes that hold them, one row at a time, the
// conversions took 78 % of the FP64 pipe: scans at N = 2e6, l_max = 16 0.089 ->
// 0.085 ms; N = 4e6, l_max = 24 0.296 -> 0.280). Bound by memory and by the
// compensated additions' issue slots.
constexpr int kTsRows = 32;    // components per CTA
constexpr int kTsTiles = 128;  // tiles per CTA

template <class T>
__global__ void __launch_bounds__(256) k_tile_scan(const T* __restrict__ agg, T* __restrict__ pfx,
                                                   double* __restrict__ gagg, double* __restrict__ csum, int64_t tw,
                                                   int64_t ts, int nc) {
  chain_wait();
  using V4 = typename Vec4<T>::type;
  using C = CSum<T>;
  __shared__ T buf[kTsRows][kTsTiles + 1];  // [row][tile], padded: the transposed reads hit distinct banks
  __shared__ C gt[kTsTiles / 32][kTsRows];  // group totals
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = lane & 7;
  const int64_t tile0 = int64_t(blockIdx.x) * kTsTiles;
  const int u0 = int(blockIdx.y) * kTsRows;
  const int64_t tile = tile0 + 4 * lane;
  V4 v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int u = u0 + 4 * warp + k;
    if (u < nc && tile < tw) {
      v[k] = *reinterpret_cast<const V4*>(agg + int64_t(u) * ts + tile);
    } else {
      v[k].x = v[k].y = v[k].z = v[k].w = T(0);
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int row = 4 * warp + k, u = u0 + row;
    if (u >= nc) break;  // warp-uniform
    V4 o;
    if (u & 1) {  // Is: exclusive suffix
      const C f2 = cs_of(v[k].w), f1 = cs_add(f2, cs_of(v[k].z)), f0 = cs_add(f1, cs_of(v[k].y)),
              sum = cs_add(f0, cs_of(v[k].x));
      C x = cs_shfl_down(sum, 1);
      if (r == 7) x = cs_of(T(0));
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) {
        const C y = cs_shfl_down(x, d);
        if (r + d < 8) x = cs_add(x, y);
      }
      o.x = cs_round(cs_add(x, f0)); o.y = cs_round(cs_add(x, f1)); o.z = cs_round(cs_add(x, f2));
      o.w = cs_round(x);
      if (r == 0) gt[lane >> 3][row] = cs_add(x, sum);
    } else {      // Rs: exclusive prefix
      const C e1 = cs_of(v[k].x), e2 = cs_add(e1, cs_of(v[k].y)), e3 = cs_add(e2, cs_of(v[k].z)),
              sum = cs_add(e3, cs_of(v[k].w));
      C x = cs_shfl_up(sum, 1);
      if (r == 0) x = cs_of(T(0));
#pragma unroll
      for (int d = 1; d < 8; d <<= 1) {
        const C y = cs_shfl_up(x, d);
        if (r >= d) x = cs_add(x, y);
      }
      o.x = cs_round(x); o.y = cs_round(cs_add(x, e1)); o.z = cs_round(cs_add(x, e2));
      o.w = cs_round(cs_add(x, e3));
      if (r == 7) gt[lane >> 3][row] = cs_add(x, sum);
    }
    buf[row][4 * lane] = o.x; buf[row][4 * lane + 1] = o.y;
    buf[row][4 * lane + 2] = o.z; buf[row][4 * lane + 3] = o.w;
  }
  __syncthreads();
  // transposed write: warp w writes tiles w, w + 8, ..., lane = row; the group totals first
  const int u = u0 + lane;
  if (u < nc) {
    if (warp < kTsTiles / 32 && tile0 + 32 * warp < tw) gagg[(tile0 / 32 + warp) * nc + u] = cs_double(gt[warp][lane]);
    if (csum && warp == kTsTiles / 32) {  // the sum of this CTA's groups
      double sum = 0.0;
      for (int k = 0; k < kTsTiles / 32 && tile0 + 32 * k < tw; ++k) sum += cs_double(gt[k][lane]);
      csum[int64_t(blockIdx.x) * nc + u] = sum;
    }
    const int tend = tw - tile0 < kTsTiles ? int(tw - tile0) : kTsTiles;
    T* dst = pfx + (tile0 + warp) * nc + u;
    const int64_t step = 8 * int64_t(nc);
#pragma unroll 4
    for (int t = warp; t < tend; t += 8, dst += step) *dst = buf[lane][t];
  }
}

// ============================================================================
// Group scan. Input: the FP64 totals gagg[g][u] of the scan groups (written
// by the tile scan). Output: gbase[g][u] = the sum over the earlier groups (Rs
// components, u even) or over the later groups (Is components, u odd), each
// summed in its own direction, and the totals tot / totd.
// The groups are cut into nseg segments of G groups (G a multiple of 8);
// CTA (column block b, segment s) handles components 32 b + lane with its 8
// warps splitting the segment. k_group_sums forms the warp and segment sums;
// the last CTA of a column block to finish (an atomic ticket, no waiting)
// scans the segment sums of that block in a fixed order, so the result is
// the same whichever CTA finishes last. k_group_bases then walks each warp's
// groups once more and writes the bases. Up to kGsOne groups one kernel
// (k_group_scan) does all of it.
// The CTA that completes the last column block (a second ticket) runs the
// step's finalize, which needs the totals alone.
// Work space w (FP64): [nseg][8][nc] warp sums, then [nseg][nc] segment sums,
// then [nseg][nc] segment bases.
// ============================================================================

// Finalize: u_asy(t_n) and its products with the drive coefficients, the kick
// weight, and Q_diff(t_n) = -(1/n~) sum over odd
// l of c_l' b^P_l * (sum_i q_i Is_l^0(x_i)) (Sec. 4; Is_l^0 = P_l(cos t)/r^{l+1}).
// By one warp (the per-degree products and loads one per lane).
__device__ __forceinline__ void finalize_step(const FinalizeArgs& a, int lane) {
  static_assert(kTabL <= 32, "one degree per lane");
  StepState* st = a.st;
  const int64_t n = st->next;
  const int32_t sync = st->sync, nabs = st->nabs_step;
  const double t = double(n) * a.dt;
  double u = 0.0;
  if (a.drive_kind == 0) {
    const double z = (t - a.t0) / a.sigma;
    u = a.v_hat * exp(-0.5 * z * z);
  } else if (a.drive_kind == 1) {
    u = n == 0 ? a.v_hat : 0.0;
  }
  if (lane < kTabL) st->drive_f[lane] = float(u * a.cdrive[lane]);
  const double is0 = (lane & 1) && lane <= a.L ? __ldcg(a.totd + 2 * (lane - 1) + 1) : 0.0;  // l = lane
  double q = 0.0;
  for (int l = 1; l <= a.L; l += 2) q += a.canti[l] * __shfl_sync(0xffffffffu, is0, l);
  q *= -a.inv_ntilde;
  if (lane != 0) return;
  st->step = n;
  st->u = u;
  const double kick = sync ? 0.5 * a.dt : a.dt;
  st->kick = kick;
  st->kick_f = float(kick);
  // electrons absorbed at the probe since the last fold (wall_rule 2) join Q_S
  // (charge -1 each) before the field of this step is evaluated
  const double qs_acc = st->qs_acc - double(nabs), qs = a.q_s + qs_acc;
  st->qs_acc = qs_acc;
  st->qs_h = float(qs);
  st->qs_l = float(qs - double(float(qs)));
  st->nabs_total += nabs;
  st->nabs_step = 0;
  if (a.record) {
    const int64_t h = n - a.first;
    if (h >= 0 && h < a.cap) {
      a.qhist[h] = q;
      a.uhist[h] = u;
    }
    st->next = n + 1;
    st->sync = 0;
  }
}

// After the totals of a block of components are written (by warp 0 of the calling CTA): the last of
// the `blocks` blocks finalizes the step.
__device__ __forceinline__ void group_finalize(const FinalizeArgs& fin, unsigned* ticket, unsigned blocks, unsigned warp,
                                               unsigned lane) {
  if (!fin.st || warp != 0) return;
  __threadfence();
  __syncwarp();
  unsigned t = 0;
  if (lane == 0) t = atomicAdd(&ticket[blocks], 1u);
  if (__shfl_sync(0xffffffffu, t, 0) == blocks - 1) {
    __threadfence();
    if (lane == 0) ticket[blocks] = 0u;
    finalize_step(fin, int(lane));
  }
}

// Up to kGsOne groups: the bases and the totals in one kernel. csum holds the sums of runs of
// kGsRun groups (of one CTA of the tile scan each; with one segment they are formed here); CTA
// (column block b, segment s) has kGsWarps runs, one per warp. The CTA adds up the runs of the other segments before it (Rs) or after it
// (Is), its warps taking them in turn; then each warp adds the segment's own runs on that side and
// walks its groups. The CTAs of the first segment form the totals. Every CTA sums up to
// kGsOne / kGsRun runs again, in FP64 (1/64 of the FP32 rate): that sets kGsOne. A step
// against sums, segment scan and bases in two kernels: N = 1e5, l_max = 16 84.6 -> 82.2 us, N = 3e5,
// l_max = 8 86.2 -> 84.1; 489 groups (N = 5e5, l_max = 1) 71.7 and 71.6, 684 (N = 7e5) 229 and 231.
constexpr int kGsRun = kTsTiles / 32;
template <class T>
__global__ void __launch_bounds__(kGsWarps * 32) k_group_scan(const double* __restrict__ gagg,
                                                              const double* __restrict__ csum, unsigned* ticket,
                                                              T* __restrict__ gbase, T* __restrict__ tot, double* totd,
                                                              int ngroups, int nc, FinalizeArgs fin) {
  chain_wait();
  __shared__ double others[kGsWarps][32], own[kGsWarps][32];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = int(blockIdx.x) * 32 + int(lane);
  const bool okc = c < nc, suffix = (c & 1) != 0, first = blockIdx.y == 0;
  const int nrun = (ngroups + kGsRun - 1) / kGsRun, r0 = int(blockIdx.y) * kGsWarps, r = r0 + int(warp);
  const int64_t g0 = int64_t(r) * kGsRun;
  double v[kGsRun];
#pragma unroll
  for (int k = 0; k < kGsRun; ++k) v[k] = okc && g0 + k < ngroups ? gagg[(g0 + k) * nc + c] : 0.0;
  double rest = 0.0;
  if (gridDim.y > 1) {
    own[warp][lane] = okc && r < nrun ? csum[int64_t(r) * nc + c] : 0.0;
    double sum = 0.0;
    // in the first segment both kinds of component take the runs after it (its bases or the totals)
#pragma unroll 4
    for (int k = int(warp); k < nrun; k += kGsWarps)
      if (okc && (suffix || first ? k >= r0 + kGsWarps : k < r0)) sum += csum[int64_t(k) * nc + c];
    others[warp][lane] = sum;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kGsWarps; ++k) rest += others[k][lane];
  } else {  // one segment: the runs summed here
    double sum = v[0];
#pragma unroll
    for (int k = 1; k < kGsRun; ++k) sum += v[k];
    own[warp][lane] = sum;
    __syncthreads();
  }
  double run = first && !suffix ? 0.0 : rest;
#pragma unroll
  for (int k = 0; k < kGsWarps; ++k)
    if (suffix ? k > int(warp) : k < int(warp)) run += own[k][lane];
#pragma unroll
  for (int q = 0; q < kGsRun; ++q) {
    const int64_t g = g0 + (suffix ? kGsRun - 1 - q : q);
    if (okc && g < ngroups) gbase[g * nc + c] = T(run);
    run += suffix ? v[kGsRun - 1 - q] : v[q];
  }
  if (!first) return;
  if (warp == 0 && okc) {
#pragma unroll
    for (int k = 0; k < kGsWarps; ++k) rest += own[k][lane];
    tot[c] = T(rest);
    totd[c] = rest;
  }
  group_finalize(fin, ticket, gridDim.x, warp, lane);
}

template <class T>
__global__ void __launch_bounds__(kGsWarps * 32) k_group_sums(const double* __restrict__ gagg,
                                                              double* __restrict__ w, unsigned* __restrict__ ticket,
                                                              T* __restrict__ tot, double* totd,
                                                              int64_t ngroups, int nc, int64_t G, int nseg,
                                                              FinalizeArgs fin) {
  chain_wait();
  __shared__ double ws[kGsWarps][32];
  __shared__ double sst[kGsMaxSeg][32];  // the segment sums of this column block (last CTA)
  __shared__ bool last;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  const bool okc = c < nc, suffix = (c & 1) != 0;
  const int seg = blockIdx.y;
  double* wsum = w;
  double* ssum = w + int64_t(kGsMaxSeg) * kGsWarps * nc;
  double* sbase = ssum + int64_t(kGsMaxSeg) * nc;
  const int64_t per = G / kGsWarps;
  const int64_t g0 = int64_t(seg) * G + warp * per;
  const int64_t g1 = g0 + per < ngroups ? g0 + per : ngroups;
  double run = 0.0;
  if (okc) {
#pragma unroll 4
    for (int64_t g = g0; g < g1; ++g) run += gagg[g * nc + c];
    wsum[(int64_t(seg) * kGsWarps + warp) * nc + c] = run;
  }
  ws[warp][lane] = run;
  __syncthreads();
  if (warp == 0 && okc) {
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < kGsWarps; ++k) sum += ws[k][lane];
    ssum[int64_t(seg) * nc + c] = sum;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&ticket[blockIdx.x], 1u) == unsigned(nseg - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  // all warps stage the segment sums (independent loads in flight together),
  // then warp 0 scans them from shared memory in a fixed order
  for (int k = int(warp); k < nseg; k += kGsWarps) sst[k][lane] = okc ? __ldcg(ssum + int64_t(k) * nc + c) : 0.0;
  __syncthreads();
  if (warp == 0 && okc) {
    double all = 0.0;
    for (int k = 0; k < nseg; ++k) {
      const int s2 = suffix ? nseg - 1 - k : k;
      sbase[int64_t(s2) * nc + c] = all;
      all += sst[s2][lane];
    }
    tot[c] = T(all);
    totd[c] = all;
  }
  if (threadIdx.x == 0) ticket[blockIdx.x] = 0u;  // ready for the next step
  group_finalize(fin, ticket, gridDim.x, warp, lane);
}

template <class T>
__global__ void __launch_bounds__(kGsWarps * 32) k_group_bases(const double* __restrict__ gagg,
                                                               const double* __restrict__ w, T* __restrict__ gbase,
                                                               int64_t ngroups, int nc, int64_t G) {
  chain_wait();
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  if (c >= nc) return;  // no barrier below
  const int seg = blockIdx.y;
  const bool suffix = (c & 1) != 0;
  const double* wsum = w;
  const double* sbase = w + int64_t(kGsMaxSeg) * (kGsWarps + 1) * nc;
  double run = sbase[int64_t(seg) * nc + c];
#pragma unroll
  for (int k = 0; k < kGsWarps; ++k)
    if (suffix ? unsigned(k) > warp : unsigned(k) < warp) run += wsum[(int64_t(seg) * kGsWarps + k) * nc + c];
  const int64_t per = G / kGsWarps;
  const int64_t g0 = int64_t(seg) * G + warp * per;
  const int64_t g1 = g0 + per < ngroups ? g0 + per : ngroups;
#pragma unroll 4
  for (int64_t k = 0; k < g1 - g0; ++k) {
    const int64_t g = suffix ? g1 - 1 - k : g0 + k;
    gbase[g * nc + c] = T(run);
    run += gagg[g * nc + c];
  }
}

template <class T>
void launch_scans(const T* agg, T* pfx, double* gagg, double* work, unsigned* ticket, T* gbase, T* tot, double* totd,
                  int64_t ntiles, int nc, int gseg, const FinalizeArgs* fin, LaunchSeq& seq) {
  const int64_t tw = tiles_whole(ntiles), ts = tile_stride(ntiles), ngroups = tw / kTilesPerGroup;
  if (tw <= 0) return;
  const bool one = ngroups <= kGsOne;
  const dim3 grid(unsigned((tw + kTsTiles - 1) / kTsTiles), unsigned((nc + kTsRows - 1) / kTsRows));
  const FinalizeArgs fa = fin ? *fin : FinalizeArgs{};
  const dim3 cols1(unsigned(gs_col_blocks(nc)), unsigned((grid.x + kGsWarps - 1) / kGsWarps));
  seq(k_tile_scan<T>, grid, 256, 0, agg, pfx, gagg, one && cols1.y > 1 ? work : nullptr, tw, ts, nc);
  if (one) {
    seq(k_group_scan<T>, cols1, kGsWarps * 32, 0, gagg, work, ticket, gbase, tot, totd, int(ngroups), nc, fa);
    return;
  }
  const int64_t G = gs_seg_len(ngroups, gseg);
  const int nseg = int(gs_nseg(ngroups, gseg));
  const dim3 cols(unsigned(gs_col_blocks(nc)), unsigned(nseg));
  seq(k_group_sums<T>, cols, kGsWarps * 32, 0, gagg, work, ticket, tot, totd, ngroups, nc, G, nseg, fa);
  seq(k_group_bases<T>, cols, kGsWarps * 32, 0, gagg, work, gbase, ngroups, nc, G);
}

// Step state after a load: step 0, nothing recorded, the first kick is a half kick.
__global__ void k_init_step(StepState* st) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  st->step = 0;
  st->next = 0;
  st->u = 0.0;
  st->kick = 0.0;
  st->sync = 1;
  st->nabs_step = 0;
  st->qs_acc = 0.0;
  st->nabs_total = 0;
}

void launch_init_step(StepState* st, cudaStream_t s) { k_init_step<<<1, 32, 0, s>>>(st); }

// ============================================================================
// Spectrum sums (FP64): sum_n x_n e^{-i w n dt} of two real series at nf
// frequencies. FP64 runs at 1/64 of the FP32 rate here, so the kernel is bound
// by its FP64 operations and by how many SMs take part: one warp per 32
// frequencies and segment of samples, the segments' partial sums added in
// order by k_dft_sum. Inside a segment the samples go in blocks of 32 around
// the block's centre c: with the pair sums s_b = x_{c+b} + x_{c-b} and
// differences d_b (formed once per block in shared memory; b = 1/2 .. 31/2)
//   sum_n x_n e^{-i w n dt} = e^{-i w c dt} sum_b (s_b cos(w b dt) - i d_b sin(w b dt)),
// one multiply-add per sample; cos and sin of the 16 offsets stay in registers
// and the centre's phase advances by one rotation per block (recomputed every
// kDftResync blocks). A segment whose samples of a series are all zero (the
// drive after its pulse) leaves that series out: exact zeros. One thread per
// frequency over all samples, with a rotation per sample, took 7.96 ms at
// ns = 20000, nf = 1000 (8 CTAs, 10 operations per sample); this form 0.092 ms and
// 0.010 ms for the sum of the segments.
// ============================================================================
constexpr int kDftBlock = 32, kDftHalf = kDftBlock / 2;
constexpr int kDftResync = 16;      // blocks between exact phases; also the blocks staged at once
constexpr int64_t kDftCtas = 1216;  // CTAs (warps) aimed at: 8 per SM
constexpr int kDftMaxSeg = 64;

// Blocks per segment and segments for ns samples at nf frequencies.
static int64_t dft_seg_blocks(int64_t ns, int64_t nf) {
  const int64_t nblk = (ns + kDftBlock - 1) / kDftBlock, cols = (nf + 31) / 32;
  int64_t nseg = (kDftCtas + cols - 1) / cols;
  if (nseg > kDftMaxSeg) nseg = kDftMaxSeg;
  const int64_t nb = (nblk + nseg - 1) / nseg;
  return nb < 4 ? 4 : nb;  // fewer would spend more on the phases than on the samples
}
static int64_t dft_segments(int64_t ns, int64_t nf) {
  const int64_t per = dft_seg_blocks(ns, nf) * kDftBlock;
  return (ns + per - 1) / per;
}
int64_t dft_work_doubles(int64_t ns, int64_t nf) { return 4 * nf * (1 + dft_segments(ns, nf)); }

__global__ void __launch_bounds__(32) k_dft(const double* __restrict__ q, const double* __restrict__ u, int64_t ns,
                                            double dt, double first_kick, int64_t nf, double w_max,
                                            int64_t seg_blocks, double* __restrict__ part) {
  __shared__ __align__(16) double2 xq[kDftResync][kDftHalf];  // (s_b, d_b) of q_n - q_0
  __shared__ __align__(16) double2 xu[kDftResync][kDftHalf];  // and of kw_n u_n
  const int lane = threadIdx.x;
  const int64_t jf = int64_t(blockIdx.x) * 32 + lane;
  const double w = double(jf + 1) * (w_max / double(nf));  // past nf: computed, not written
  const double th = w * dt;
  double c[kDftHalf], s[kDftHalf];  // cos, sin of th (b + 1/2)
  sincos(0.5 * th, &s[0], &c[0]);
  {
    const double rc = 1.0 - 2.0 * s[0] * s[0], rs = 2.0 * s[0] * c[0];
#pragma unroll
    for (int b = 1; b < kDftHalf; ++b) {
      c[b] = c[b - 1] * rc - s[b - 1] * rs;
      s[b] = s[b - 1] * rc + c[b - 1] * rs;
    }
  }
  double br, bi;  // rotation by one block
  sincos(th * double(kDftBlock), &bi, &br);
  const double q0 = q[0];
  const int64_t a0 = int64_t(blockIdx.y) * seg_blocks;
  const int64_t nblk = (ns + kDftBlock - 1) / kDftBlock;
  const int64_t a1 = a0 + seg_blocks < nblk ? a0 + seg_blocks : nblk;
  double Qr = 0, Qi = 0, Ur = 0, Ui = 0;
  for (int64_t a = a0; a < a1; a += kDftResync) {
    const int nb = a1 - a < kDftResync ? int(a1 - a) : kDftResync;
    bool anyq = false, anyu = false;
    __syncwarp();
    for (int k = lane; k < nb * kDftHalf; k += 32) {
      const int blk = k / kDftHalf, b = k % kDftHalf;
      const int64_t hi = (a + blk) * kDftBlock + kDftHalf + b, lo = (a + blk) * kDftBlock + kDftHalf - 1 - b;
      const double qh = hi < ns ? q[hi] - q0 : 0.0, ql = lo < ns ? q[lo] - q0 : 0.0;
      const double uh = hi < ns ? dt * u[hi] : 0.0;  // hi >= 16: never the first step
      const double ul = lo < ns ? (lo == 0 ? first_kick : dt) * u[lo] : 0.0;
      xq[blk][b] = make_double2(qh + ql, qh - ql);
      xu[blk][b] = make_double2(uh + ul, uh - ul);
      anyq = anyq || qh != 0.0 || ql != 0.0;  // true for NaN
      anyu = anyu || uh != 0.0 || ul != 0.0;
    }
    anyq = __any_sync(0xffffffffu, anyq);
    anyu = __any_sync(0xffffffffu, anyu);
    __syncwarp();
    double pr, pi;  // e^{-i w c dt} of the block's centre
    sincos(th * (double(a * kDftBlock) + (kDftHalf - 0.5)), &pi, &pr);
    pi = -pi;
    for (int blk = 0; blk < nb; ++blk) {
      if (anyq) {
        double A = 0, B = 0;
#pragma unroll
        for (int b = 0; b < kDftHalf; ++b) {
          const double2 x = xq[blk][b];
          A = fma(x.x, c[b], A);
          B = fma(-x.y, s[b], B);
        }
        Qr += pr * A - pi * B;
        Qi += pr * B + pi * A;
      }
      if (anyu) {
        double A = 0, B = 0;
#pragma unroll
        for (int b = 0; b < kDftHalf; ++b) {
          const double2 x = xu[blk][b];
          A = fma(x.x, c[b], A);
          B = fma(-x.y, s[b], B);
        }
        Ur += pr * A - pi * B;
        Ui += pr * B + pi * A;
      }
      const double npr = pr * br + pi * bi;
      pi = pi * br - pr * bi;
      pr = npr;
    }
  }
  if (jf < nf) {
    double* o = part + 4 * (int64_t(blockIdx.y) * nf + jf);
    o[0] = Qr; o[1] = Qi; o[2] = Ur; o[3] = Ui;
  }
}

// out[jf] = the segments' sums in order, Q scaled by dt: one thread per value.
__global__ void __launch_bounds__(128) k_dft_sum(const double* __restrict__ part, int64_t nseg, int64_t nf, double dt,
                                                 double* __restrict__ out) {
  const int64_t k = int64_t(blockIdx.x) * 128 + threadIdx.x;
  if (k >= 4 * nf) return;
  double v = 0.0;
#pragma unroll 8
  for (int64_t g = 0; g < nseg; ++g) v += part[g * 4 * nf + k];
  out[k] = (k & 3) < 2 ? dt * v : v;
}

void launch_dft(const double* q, const double* u, int64_t ns, double dt, double first_kick, int64_t nf,
                double w_max, double* work, cudaStream_t s) {
  const int64_t nseg = dft_segments(ns, nf);
  const dim3 grid(unsigned((nf + 31) / 32), unsigned(nseg));
  double* part = work + 4 * nf;
  k_dft<<<grid, 32, 0, s>>>(q, u, ns, dt, first_kick, nf, w_max, dft_seg_blocks(ns, nf), part);
  k_dft_sum<<<unsigned((4 * nf + 127) / 128), 128, 0, s>>>(part, nseg, nf, dt, work);
}

template <class T> cudaError_t preload_core_kernels_t() {
  cudaFuncAttributes fa;
  const void* fns[] = {
      reinterpret_cast<const void*>(&k_reorder<T>),     reinterpret_cast<const void*>(&k_keys<T>),
      reinterpret_cast<const void*>(&k_load<T>),        reinterpret_cast<const void*>(&k_state_dump<T>),
      reinterpret_cast<const void*>(&k_scatter_by_id<T>), reinterpret_cast<const void*>(&k_state_out<T>),
      reinterpret_cast<const void*>(&k_tile_scan<T>),   reinterpret_cast<const void*>(&k_group_sums<T>),
      reinterpret_cast<const void*>(&k_group_bases<T>), reinterpret_cast<const void*>(&k_group_scan<T>)};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t preload_core_kernels() {
  if (set_sort_attributes() != cudaSuccess) return cudaErrorInvalidValue;
  cudaFuncAttributes fa;
  const void* fns[] = {reinterpret_cast<const void*>(&k_sort_hist),
                       reinterpret_cast<const void*>(&k_sort_rowscan),
                       reinterpret_cast<const void*>(&k_sort_scatter),
                       reinterpret_cast<const void*>(&k_sort_count),
                       reinterpret_cast<const void*>(&k_sort_spread),
                       reinterpret_cast<const void*>(&k_bucket_sort<float, kBsOneThreads, 1>),
                       reinterpret_cast<const void*>(&k_bucket_sort<double, kBsOneThreads, 1>),
                       reinterpret_cast<const void*>(&k_bucket_sort<float, kBsThreads, kBsPerSM>),
                       reinterpret_cast<const void*>(&k_bucket_sort<double, kBsThreads, kBsPerSM>),
                       reinterpret_cast<const void*>(&k_init_step)};
  for (const void* f : fns) {
    const cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
  }
  const cudaError_t e = preload_core_kernels_t<float>();
  return e != cudaSuccess ? e : preload_core_kernels_t<double>();
}

// explicit instantiations
#define IMRP_INST_CORE(T)                                                                          \
  template const uint32_t* launch_radix_sort<T>(uint32_t*, uint32_t*, uint32_t*, uint32_t*, void*, int64_t, int,      \
                                                const Part<T>*, T* const*, uint32_t*, int*, LaunchSeq&, bool);       \
  template void launch_reorder<T>(const Part<T>*, T* const*, uint32_t*, const uint32_t*, int64_t,  \
                                  LaunchSeq&);                                                     \
  template void launch_keys<T>(const Part<T>*, uint32_t*, uint32_t*, int64_t, double, LaunchSeq&); \
  template void launch_load<T>(const double*, const double*, const uint32_t*, Part<T>*, uint32_t*, \
                               uint32_t*, int64_t, double, int*, cudaStream_t);                    \
  template void launch_state_dump<T>(const Part<T>*, double*, double*, uint32_t*, int64_t,         \
                                     cudaStream_t);                                                \
  template void launch_scatter_by_id<T>(const T* const*, int, const uint32_t*, double*, int64_t,   \
                                        LaunchSeq&);                                               \
  template void launch_state_out<T>(const Part<T>*, double*, double*, uint32_t*, int64_t, cudaStream_t); \
  template void launch_scans<T>(const T*, T*, double*, double*, unsigned*, T*, T*, double*, int64_t, int, int, \
                                const FinalizeArgs*, LaunchSeq&);
IMRP_INST_CORE(float)
IMRP_INST_CORE(double)

}  // namespace imrp
