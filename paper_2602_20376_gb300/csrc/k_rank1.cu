// k_rank1.cu -- exact rank-1 solver by an angular sweep (Sec. 2.5,
// Algorithm 1), and the same sweep scored on a graph's exact cut.
//
// For Q = q q^H the objective of z(c) with c = exp(i phi) is |q^H z|^2.  As
// phi runs over one period 2 pi / K, every coordinate's rounded code
// advances exactly once, at the angle where arg(q_i) + phi crosses a
// decision boundary (Sec. 2.5: the optimum is one of these n + 1 states).
// Convention (shared with the oracle): t_i = K arg(q_i) / (2 pi), the start
// code is floor(t_i) mod K and coordinate i advances at
// phi_i = (2 pi / K)(1/2 + floor(t_i) - t_i); states are the prefixes of the
// coordinates sorted by (phi_i, i).
//
// GPU steps: per-coordinate key (FP64), a stable sort of (key, index) pairs
// (a bitonic network, or radix passes over eight 8-bit digits), the
// increments conj(q_i) w^{k_i} (w - 1) in sorted order, an FP64 prefix scan
// giving q^H z for every state, and the argmax (ties to the earliest state).
// With a CSR graph the state at which coordinate i advances changes the cut by
// the sum over i's neighbours (each edge is stored in both rows), so one pass
// over the rows gives every state's change and an int64 prefix scan its exact
// cut (Max-K-Cut reading of Sec. 1).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <utility>

#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

constexpr int kR1Threads = 256;
constexpr int kR1Local = 2048;  // elements sorted per block in shared memory
// Up to here the sort is the bitonic network, radix passes above.  A radix pass
// costs three launches whatever n is, and below some 10^5 pairs they do little
// but wait; the network's launches grow with log^2 n (1 up to 2048 pairs, 4 at
// 4096, 28 at 2^17).  Whole sweep with a graph, network / radix passes: n = 3000
// 186 / 315 us, 16384 230 / 345, 65536 304 / 357, 80000 346 / 365, 131072 359 /
// 378; at 2^18 the network would take 37 launches over twice the pairs.
constexpr int64_t kR1Bitonic = 1 << 17;
constexpr int kR1Scan = 2048;   // elements per block in the scans (8 a thread)
constexpr int kR1BaseBlocks = 1024;  // blocks that leave a partial of the base sum (at most)
// radix sort: a block takes kR1Tile consecutive pairs, a warp 32 at a time of
// its own consecutive share
constexpr int kR1SortThreads = 256;
constexpr int kR1PerThread = 16;
constexpr int kR1Tile = kR1SortThreads * kR1PerThread;
constexpr int kR1Digits = 256;
static_assert(kR1SortThreads == kR1Digits, "a thread per digit");
constexpr int kR1SortSmem = kR1Tile * 12 + (kR1SortThreads / 32) * kR1Digits * 4;

struct R1Tables {
  double zr[kMaxK], zi[kMaxK];
};

// order-preserving map of a double to uint64
__device__ __forceinline__ uint64_t r1_key(double x) {
  const uint64_t b = static_cast<uint64_t>(__double_as_longlong(x));
  return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}

// Whether this block is the last of the grid to arrive (the counter returns
// to zero); the other blocks' global writes are then visible to it.
__device__ __forceinline__ bool r1_last_block(unsigned* counter) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(counter, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last != 0;
}

// Keys, start codes, and S0 = sum_i conj(q_i) w^{code0_i} (block sums, added
// by the last block in a fixed order).  Entries n..npad-1 sort last.  Bound:
// FP64 (atan2).
__global__ void __launch_bounds__(kR1Threads) r1_prep_kernel(const double2* __restrict__ q, int64_t n, int64_t npad,
                                                             int K, const __grid_constant__ R1Tables tb,
                                                             uint64_t* __restrict__ key, uint32_t* __restrict__ idx,
                                                             uint8_t* __restrict__ code0, double2* __restrict__ part,
                                                             unsigned* counter, double2* __restrict__ s0,
                                                             int32_t* status) {
  __shared__ double2 red[kR1Threads / 32];
  auto block_sum = [&](double2 v) {  // meaningful in thread 0
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, m);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, m);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    for (int k = 1; k < kR1Threads / 32; ++k) {
      v.x += red[k].x;
      v.y += red[k].y;
    }
    return v;
  };
  double2 s = make_double2(0.0, 0.0);
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kR1Threads + threadIdx.x; i < npad;
       i += static_cast<int64_t>(gridDim.x) * kR1Threads) {
    idx[i] = i >= n ? 0xFFFFFFFFu : static_cast<uint32_t>(i);
    if (i >= n) {
      key[i] = ~0ull;
      continue;
    }
    const double2 v = q[i];
    if (!isfinite(v.x) || !isfinite(v.y)) dev_fail(status, LRQ_EINVAL);
    const double th = atan2(v.y, v.x);
    const double t = static_cast<double>(K) * th / (2.0 * kPi);
    const double fl = floor(t);
    const double phi = (2.0 * kPi / static_cast<double>(K)) * (0.5 + fl - t);
    long long kk = static_cast<long long>(fl) % K;
    if (kk < 0) kk += K;
    key[i] = r1_key(phi);
    code0[i] = static_cast<uint8_t>(kk);
    s.x += v.x * tb.zr[kk] + v.y * tb.zi[kk];
    s.y += v.x * tb.zi[kk] - v.y * tb.zr[kk];
  }
  s = block_sum(s);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
  if (!r1_last_block(counter)) return;
  s = make_double2(0.0, 0.0);
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += kR1Threads) {
    const double2 o = __ldcg(part + b);
    s.x += o.x;
    s.y += o.y;
  }
  s = block_sum(s);
  if (threadIdx.x == 0) *s0 = s;
}

__device__ __forceinline__ bool r1_less(uint64_t ka, uint32_t ia, uint64_t kb, uint32_t ib) {
  return ka < kb || (ka == kb && ia < ib);
}

// n <= kR1Bitonic: a bitonic network over the pairs, padded to a power of two.
// Stages with partner distance below kR1Local run in shared memory: a block
// owns kR1Local consecutive pairs and takes the merge sizes k_first..k_last (all
// up to kR1Local in the first launch, then the tail of one size each).
__global__ void __launch_bounds__(kR1Local / 2) r1_sort_local(uint64_t* __restrict__ key, uint32_t* __restrict__ idx,
                                                              int k_first, int k_last) {
  __shared__ uint64_t sk[kR1Local];
  __shared__ uint32_t si[kR1Local];
  const int base = static_cast<int>(blockIdx.x) * kR1Local;  // below kR1Bitonic
  for (int t = threadIdx.x; t < kR1Local; t += blockDim.x) {
    sk[t] = key[base + t];
    si[t] = idx[base + t];
  }
  __syncthreads();
  for (int k = k_first; k <= k_last; k <<= 1) {
    for (int j = min(k >> 1, kR1Local / 2); j > 0; j >>= 1) {
      const int t = threadIdx.x;
      const int a = (t / j) * 2 * j + (t % j);
      const int b = a + j;
      const bool up = ((base + a) & k) == 0;
      const bool sw = up ? r1_less(sk[b], si[b], sk[a], si[a]) : r1_less(sk[a], si[a], sk[b], si[b]);
      if (sw) {
        const uint64_t tk = sk[a];
        sk[a] = sk[b];
        sk[b] = tk;
        const uint32_t ti = si[a];
        si[a] = si[b];
        si[b] = ti;
      }
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < kR1Local; t += blockDim.x) {
    key[base + t] = sk[t];
    idx[base + t] = si[t];
  }
}

// one stage (merge size k, partner distance j >= kR1Local) in global memory, a
// thread per pair of pairs
__global__ void __launch_bounds__(kR1Threads) r1_sort_global(uint64_t* __restrict__ key, uint32_t* __restrict__ idx,
                                                             int npad, int k, int j) {
  const int t = static_cast<int>(blockIdx.x) * kR1Threads + threadIdx.x;
  if (t >= npad / 2) return;
  const int a = (t / j) * 2 * j + (t % j), b = a + j;
  const bool up = (a & k) == 0;
  const uint64_t ka = key[a], kb = key[b];
  const uint32_t ia = idx[a], ib = idx[b];
  if (up ? r1_less(kb, ib, ka, ia) : r1_less(ka, ia, kb, ib)) {
    key[a] = kb;
    key[b] = ka;
    idx[a] = ib;
    idx[b] = ia;
  }
}

// Larger n: least-significant-digit radix sort, eight passes of 8 bits over
// the 64-bit keys, three launches each; every pass keeps the order of equal
// digits, so equal keys stay in index order.  The pairs (12 MB at n = 10^6)
// stay in L2; a pass is bound by launch latency and its reads and writes.
// n = 10^6: 213 us (scatter 15, counts 10, offsets 2 a pass); the network's 55
// launches over 2^20 padded pairs took 503.
//
// r1_hist_kernel: counts[digit][block]
__global__ void __launch_bounds__(kR1SortThreads) r1_hist_kernel(const uint64_t* __restrict__ key, int64_t n,
                                                                 int shift, uint32_t* __restrict__ counts) {
  __shared__ uint32_t hist[kR1Digits];
  hist[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kR1Tile;
#pragma unroll
  for (int u = 0; u < kR1PerThread; ++u) {
    const int64_t i = base + u * kR1SortThreads + threadIdx.x;
    // lanes with the same digit add once: skewed keys would serialise
    const int d = i < n ? static_cast<int>((key[i] >> shift) & (kR1Digits - 1)) : -1;
    const unsigned same = __match_any_sync(0xffffffffu, d);
    if (d >= 0 && (same & ((1u << (threadIdx.x & 31)) - 1u)) == 0) atomicAdd(&hist[d], __popc(same));
  }
  __syncthreads();
  counts[static_cast<int64_t>(threadIdx.x) * gridDim.x + blockIdx.x] = hist[threadIdx.x];
}

// exclusive prefix of 32 lanes' values
__device__ __forceinline__ uint32_t r1_warp_exclusive(uint32_t v, uint32_t* total) {
  const int lane = threadIdx.x & 31;
  uint32_t inc = v;
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, inc, m);
    if (lane >= m) inc += o;
  }
  *total = __shfl_sync(0xffffffffu, inc, 31);
  return inc - v;
}

// exclusive prefix of one value per thread over a block of kR1SortThreads
__device__ __forceinline__ uint32_t r1_sort_exclusive(uint32_t v, uint32_t* total) {
  __shared__ uint32_t ws[kR1SortThreads / 32];
  uint32_t t;
  uint32_t ex = r1_warp_exclusive(v, &t);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
  __syncthreads();
  t = 0;
  for (int w = 0; w < kR1SortThreads / 32; ++w) {
    if (w == static_cast<int>(threadIdx.x >> 5)) ex += t;
    t += ws[w];
  }
  __syncthreads();
  *total = t;
  return ex;
}

// a block per digit: the blocks' counts of the digit become offsets from the
// digit's first place, total[digit] their sum
__global__ void __launch_bounds__(kR1SortThreads) r1_offsets_kernel(uint32_t* __restrict__ counts, int64_t nb,
                                                                    uint32_t* __restrict__ total) {
  uint32_t* row = counts + static_cast<int64_t>(blockIdx.x) * nb;
  uint32_t carry = 0;
  for (int64_t b0 = 0; b0 < nb; b0 += kR1SortThreads) {
    const int64_t b = b0 + threadIdx.x;
    uint32_t t;
    const uint32_t ex = r1_sort_exclusive(b < nb ? row[b] : 0, &t);
    if (b < nb) row[b] = carry + ex;
    carry += t;
  }
  if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// r1_scatter_kernel: the block sorts its tile by the digit in shared memory (a
// pair's place is its digit's first place in the tile, plus the earlier warps'
// pairs of that digit, plus its rank in its warp), then writes it out in that
// order, so that a digit's pairs go to consecutive places
__global__ void __launch_bounds__(kR1SortThreads) r1_scatter_kernel(const uint64_t* __restrict__ key,
                                                                    const uint32_t* __restrict__ idx, int64_t n,
                                                                    int shift, const uint32_t* __restrict__ offs,
                                                                    const uint32_t* __restrict__ total,
                                                                    uint64_t* __restrict__ key2,
                                                                    uint32_t* __restrict__ idx2) {
  constexpr int W = kR1SortThreads / 32;
  extern __shared__ __align__(16) uint8_t r1_smem[];
  uint64_t* sk = reinterpret_cast<uint64_t*>(r1_smem);
  uint32_t* si = reinterpret_cast<uint32_t*>(sk + kR1Tile);
  uint32_t(*cnt)[kR1Digits] = reinterpret_cast<uint32_t(*)[kR1Digits]>(si + kR1Tile);
  __shared__ uint32_t place[kR1Digits];  // global place of tile position 0, as seen by the digit
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int w = 0; w < W; ++w) cnt[w][threadIdx.x] = 0;
  __syncthreads();
  const int64_t tile0 = static_cast<int64_t>(blockIdx.x) * kR1Tile;
  const int64_t base = tile0 + warp * 32 * kR1PerThread + lane;
  uint64_t k[kR1PerThread];
  uint32_t id[kR1PerThread], rank[kR1PerThread];
#pragma unroll
  for (int u = 0; u < kR1PerThread; ++u) {
    const int64_t i = base + u * 32;
    k[u] = i < n ? key[i] : 0;
    id[u] = i < n ? idx[i] : 0;
  }
#pragma unroll
  for (int u = 0; u < kR1PerThread; ++u) {
    const bool in = base + u * 32 < n;
    const int d = in ? static_cast<int>((k[u] >> shift) & (kR1Digits - 1)) : -1;
    const unsigned same = __match_any_sync(0xffffffffu, d);
    const unsigned below = same & ((1u << lane) - 1u);
    const uint32_t before = in ? cnt[warp][d] : 0;
    __syncwarp();
    if (in && below == 0) cnt[warp][d] = before + __popc(same);
    __syncwarp();
    rank[u] = before + __popc(below);
  }
  __syncthreads();
  {
    const int d = threadIdx.x;
    uint32_t c = 0, t;
    for (int w = 0; w < W; ++w) c += cnt[w][d];
    uint32_t off = r1_sort_exclusive(c, &t);  // the digit's first place in the tile
    const uint32_t digit0 = r1_sort_exclusive(total[d], &t);
    place[d] = digit0 + offs[static_cast<int64_t>(d) * gridDim.x + blockIdx.x] - off;
    for (int w = 0; w < W; ++w) {
      const uint32_t v = cnt[w][d];
      cnt[w][d] = off;
      off += v;
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kR1PerThread; ++u) {
    if (base + u * 32 < n) {
      const uint32_t at = cnt[warp][(k[u] >> shift) & (kR1Digits - 1)] + rank[u];
      sk[at] = k[u];
      si[at] = id[u];
    }
  }
  __syncthreads();
  const int rows = static_cast<int>(min(static_cast<int64_t>(kR1Tile), n - tile0));
#pragma unroll 4
  for (int p = threadIdx.x; p < rows; p += kR1SortThreads) {
    const uint64_t kk = sk[p];
    const uint32_t at = place[(kk >> shift) & (kR1Digits - 1)] + p;
    key2[at] = kk;
    idx2[at] = si[p];
  }
}

// ---- inclusive scans in two passes: block scans with block totals (whose
// exclusive prefix the last block leaves), then one pass that adds the
// offsets on the fly and takes the argmax.  Eight consecutive elements a
// thread, so that an element costs about three additions (an FP64 addition of
// a warp holds the SM's two-lane FP64 unit for 16 cycles); a doubling scan of
// 1024 elements in shared memory cost ten.
template <typename T>
__device__ __forceinline__ T r1_add(T a, T b);
template <>
__device__ __forceinline__ double2 r1_add<double2>(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
template <>
__device__ __forceinline__ long long r1_add<long long>(long long a, long long b) {
  return a + b;
}
template <typename T>
__device__ __forceinline__ T r1_zero();
template <>
__device__ __forceinline__ double2 r1_zero<double2>() {
  return make_double2(0.0, 0.0);
}
template <>
__device__ __forceinline__ long long r1_zero<long long>() {
  return 0;
}
__device__ __forceinline__ double2 r1_shfl_up(double2 v, int m) {
  return make_double2(__shfl_up_sync(0xffffffffu, v.x, m), __shfl_up_sync(0xffffffffu, v.y, m));
}
__device__ __forceinline__ long long r1_shfl_up(long long v, int m) { return __shfl_up_sync(0xffffffffu, v, m); }
__device__ __forceinline__ double2 r1_ldcg(const double2* p) { return __ldcg(p); }
__device__ __forceinline__ long long r1_ldcg(const long long* p) { return __ldcg(p); }

// exclusive prefix of one value per thread over the block, and its total
template <typename T>
__device__ __forceinline__ T r1_block_exclusive(T v, T* total) {
  __shared__ T ws[kR1Threads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T inc = v;
#pragma unroll
  for (int m = 1; m < 32; m <<= 1) {
    const T o = r1_shfl_up(inc, m);
    if (lane >= m) inc = r1_add<T>(o, inc);
  }
  if (lane == 31) ws[warp] = inc;
  T ex = r1_shfl_up(inc, 1);
  if (lane == 0) ex = r1_zero<T>();
  __syncthreads();
  T off = r1_zero<T>(), t = r1_zero<T>();
  for (int w = 0; w < kR1Threads / 32; ++w) {
    if (w == warp) off = t;
    t = r1_add<T>(t, ws[w]);
  }
  __syncthreads();
  *total = t;
  return r1_add<T>(off, ex);
}

// the elements' inclusive prefix within their block into x, and the blocks'
// exclusive prefix into sums
template <typename T>
__device__ __forceinline__ void r1_scan_tail(T (&v)[kR1Scan / kR1Threads], T* __restrict__ x, int64_t n,
                                             T* __restrict__ sums, unsigned* counter) {
  constexpr int U = kR1Scan / kR1Threads;
#pragma unroll
  for (int u = 1; u < U; ++u) v[u] = r1_add<T>(v[u - 1], v[u]);
  T total;
  const T off = r1_block_exclusive<T>(v[U - 1], &total);
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kR1Scan + static_cast<int64_t>(threadIdx.x) * U;
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (i0 + u < n) x[i0 + u] = r1_add<T>(off, v[u]);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
  if (!r1_last_block(counter)) return;
  const int64_t nb = gridDim.x, per = ceil_div(nb, kR1Threads);
  const int64_t b0 = min(nb, threadIdx.x * per), b1 = min(nb, b0 + per);
  T s = r1_zero<T>();
  for (int64_t b = b0; b < b1; ++b) s = r1_add<T>(s, r1_ldcg(sums + b));
  T off2 = r1_block_exclusive<T>(s, &total);
  for (int64_t b = b0; b < b1; ++b) {
    const T t = r1_ldcg(sums + b);
    sums[b] = off2;
    off2 = r1_add<T>(off2, t);
  }
}

// the increments of q^H z in sorted order, d_l = conj(q_i) w^{k_i} (w - 1),
// scanned as they are formed, and every coordinate's (start code, rank) in one
// word for the passes that gather both
__global__ void __launch_bounds__(kR1Threads) r1_delta_scan_kernel(
    const double2* __restrict__ q, int64_t n, int K, const uint32_t* __restrict__ idx,
    const uint8_t* __restrict__ code0, const __grid_constant__ R1Tables tb, double2* __restrict__ x,
    uint2* __restrict__ code_rank, double2* __restrict__ sums, unsigned* counter) {
  constexpr int U = kR1Scan / kR1Threads;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kR1Scan + static_cast<int64_t>(threadIdx.x) * U;
  double2 v[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t l = i0 + u;
    v[u] = make_double2(0.0, 0.0);
    if (l < n) {
      const uint32_t i = idx[l];
      const double2 w = q[i];
      const int c = code0[i], c1 = c + 1 == K ? 0 : c + 1;
      code_rank[i] = make_uint2(static_cast<uint32_t>(c), static_cast<uint32_t>(l));
      const double dzr = tb.zr[c1] - tb.zr[c], dzi = tb.zi[c1] - tb.zi[c];
      // conj(w) * dz
      v[u] = make_double2(w.x * dzr + w.y * dzi, w.x * dzi - w.y * dzr);
    }
  }
  r1_scan_tail<double2>(v, x, n, sums, counter);
}

__global__ void __launch_bounds__(kR1Threads) r1_scan_kernel(long long* __restrict__ x, int64_t n,
                                                             long long* __restrict__ sums, unsigned* counter) {
  constexpr int U = kR1Scan / kR1Threads;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * kR1Scan + static_cast<int64_t>(threadIdx.x) * U;
  long long v[U];
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = i0 + u < n ? x[i0 + u] : 0;
  r1_scan_tail<long long>(v, x, n, sums, counter);
}

// The block's largest value with the smallest state among equals, into
// bv / bs; the last block reduces the blocks' (thread 0 gets the result and
// true).  Values are integers: cuts, or the bits of non-negative doubles,
// which order alike (FP64 comparisons would run on the FP64 unit).
__device__ __forceinline__ void r1_better(long long& v, long long& st, long long o, long long os) {
  if (o > v || (o == v && os < st)) {
    v = o;
    st = os;
  }
}

__device__ __forceinline__ bool r1_best_reduce(long long v, long long st, long long* __restrict__ bv,
                                               long long* __restrict__ bs, unsigned* counter, long long* out_v,
                                               long long* out_s) {
  __shared__ long long rv[kR1Threads / 32], rs[kR1Threads / 32];
  auto reduce = [&]() {  // meaningful in thread 0
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) {
      const long long o = __shfl_xor_sync(0xffffffffu, v, m), os = __shfl_xor_sync(0xffffffffu, st, m);
      r1_better(v, st, o, os);
    }
    if ((threadIdx.x & 31) == 0) {
      rv[threadIdx.x >> 5] = v;
      rs[threadIdx.x >> 5] = st;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int k = 1; k < kR1Threads / 32; ++k) r1_better(v, st, rv[k], rs[k]);
  };
  reduce();
  if (threadIdx.x == 0) {
    bv[blockIdx.x] = v;
    bs[blockIdx.x] = st;
  }
  if (!r1_last_block(counter)) return false;
  v = -1;
  st = 0x7fffffffffffffffll;
  for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += kR1Threads) r1_better(v, st, __ldcg(bv + b), __ldcg(bs + b));
  reduce();
  *out_v = v;
  *out_s = st;
  return threadIdx.x == 0;
}

// f of states 0..n (state l + 1 = prefix l inclusive) and the argmax, ties to
// the earliest state.  One block did this alone in 1457 us at n = 10^6; now 19.
__global__ void __launch_bounds__(kR1Threads) r1_best_kernel(const double2* __restrict__ pref, int64_t n,
                                                             const double2* __restrict__ sums,
                                                             const double2* __restrict__ s0p,
                                                             long long* __restrict__ bv, long long* __restrict__ bs,
                                                             unsigned* counter, int64_t* __restrict__ best_state,
                                                             double* __restrict__ best_f) {
  const double2 s0 = *s0p;
  auto bits = [](double f) { return isnan(f) ? -1ll : __double_as_longlong(f); };
  long long f = -1, st = 0x7fffffffffffffffll;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    f = bits(s0.x * s0.x + s0.y * s0.y);
    st = 0;
  }
  for (int64_t l = static_cast<int64_t>(blockIdx.x) * kR1Threads + threadIdx.x; l < n;
       l += static_cast<int64_t>(gridDim.x) * kR1Threads) {
    const double2 p = r1_add<double2>(pref[l], sums[l / kR1Scan]);
    const double x = s0.x + p.x, y = s0.y + p.y;
    const long long g = bits(x * x + y * y);
    if (g > f) {
      f = g;
      st = l + 1;
    }
  }
  long long of, os;
  if (r1_best_reduce(f, st, bv, bs, counter, &of, &os)) {
    *best_state = os == 0x7fffffffffffffffll ? 0 : os;
    *best_f = of < 0 ? -1.0 : __longlong_as_double(of);
  }
}

// codes of state s: coordinates of rank < s have advanced by one
__global__ void r1_codes_kernel(const uint2* __restrict__ code_rank, int64_t n, int K,
                                const int64_t* __restrict__ state, uint8_t* __restrict__ z) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t s = *state;
  const uint2 cr = code_rank[i];
  const uint32_t c = cr.x + (static_cast<int64_t>(cr.y) < s ? 1u : 0u);
  z[i] = static_cast<uint8_t>(c == static_cast<uint32_t>(K) ? 0u : c);
}

// The cut of state 0 (edges counted from their lower end) into cut0, and for
// every coordinate the change of the cut at the state where it advances:
// diff[rank + 1] = sum over its edges of (cut after - cut before), the other
// end advanced already if its rank is smaller.  Each edge is in both rows, so
// no two rows write the same place; the first version had every edge add to
// two places with 64-bit atomics (245 us at n = 10^6, 3.3 * 10^6 edges; now 40).
// Bound: the gathers of the neighbours' (code, rank), one 8-byte read each.
// A thread takes a row of up to kR1RowMax entries, four gathers in flight; the
// warp takes longer rows together.
constexpr int kR1RowMax = 64;

struct R1Edge {
  int ci;
  uint32_t ri;
  long long sum;
  unsigned long long local;
};

__device__ __forceinline__ void r1_edge_one(R1Edge& a, int64_t i, int64_t j, uint2 o, int K) {
  const int cj = static_cast<int>(o.x);
  int before, after;  // the ends' code difference before and after i advances, as "equal or not"
  const int cj1 = cj + 1 == K ? 0 : cj + 1, ci1 = a.ci + 1 == K ? 0 : a.ci + 1;
  const int cjn = o.y < a.ri ? cj1 : cj;
  before = cjn != a.ci;
  after = cjn != ci1;
  a.sum += after - before;
  if (j > i && cj != a.ci) a.local += 1ull;
}

__global__ void __launch_bounds__(kR1Threads) r1_edge_kernel(const int32_t* __restrict__ rowptr,
                                                             const int32_t* __restrict__ colidx, int64_t n,
                                                             int64_t nnz, int K, const uint2* __restrict__ code_rank,
                                                             long long* __restrict__ diff,
                                                             unsigned long long* __restrict__ cut0) {
  const int lane = threadIdx.x & 31;
  unsigned long long local = 0;
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * kR1Threads + (threadIdx.x & ~31); i0 < n;
       i0 += static_cast<int64_t>(gridDim.x) * kR1Threads) {  // warp-uniform
    const int64_t i = i0 + lane;
    int64_t e0 = 0, e1 = 0;
    R1Edge a{0, 0u, 0, 0};
    if (i < n) {
      e0 = rowptr[i], e1 = rowptr[i + 1];  // bounds-guarded (a malformed CSR reads nothing outside)
      e0 = e0 < 0 ? 0 : (e0 > nnz ? nnz : e0);
      e1 = e1 < e0 ? e0 : (e1 > nnz ? nnz : e1);
      const uint2 me = code_rank[i];
      a.ci = static_cast<int>(me.x);
      a.ri = me.y;
    }
    if (e1 - e0 <= kR1RowMax) {
      for (int64_t e = e0; e < e1; e += 4) {
        int64_t j[4];
        uint2 o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          j[u] = e + u < e1 ? colidx[e + u] : -1;
          if (j[u] == i || j[u] >= n) j[u] = -1;
          o[u] = j[u] >= 0 ? code_rank[j[u]] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j[u] >= 0) r1_edge_one(a, i, j[u], o[u], K);
      }
    }
    for (unsigned big = __ballot_sync(0xffffffffu, e1 - e0 > kR1RowMax); big; big &= big - 1) {
      const int src = __ffs(big) - 1;
      const int64_t ib = i0 + src, b0 = __shfl_sync(0xffffffffu, e0, src), b1 = __shfl_sync(0xffffffffu, e1, src);
      R1Edge w{__shfl_sync(0xffffffffu, a.ci, src), __shfl_sync(0xffffffffu, a.ri, src), 0, 0};
      for (int64_t e = b0 + lane; e < b1; e += 32) {
        const int64_t j = colidx[e];
        if (j >= 0 && j < n && j != ib) r1_edge_one(w, ib, j, code_rank[j], K);
      }
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) w.sum += __shfl_xor_sync(0xffffffffu, w.sum, m);
      local += w.local;
      if (lane == src) a.sum = w.sum;
    }
    local += a.local;
    if (i < n) diff[static_cast<int64_t>(a.ri) + 1] = a.sum;
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) local += __shfl_xor_sync(0xffffffffu, local, m);
  if (lane == 0 && local) atomicAdd(cut0, local);
}

// the best state by cut (ties to the earliest); pref and sums hold the scan
__global__ void __launch_bounds__(kR1Threads) r1_best_cut_kernel(const long long* __restrict__ pref, int64_t n,
                                                                 const long long* __restrict__ sums,
                                                                 const unsigned long long* __restrict__ cut0,
                                                                 long long* __restrict__ bv, long long* __restrict__ bs,
                                                                 unsigned* counter, int64_t* __restrict__ best_state,
                                                                 int64_t* __restrict__ best_cut) {
  const long long c0 = static_cast<long long>(*cut0);
  long long c = -1, st = 0x7fffffffffffffffll;
  for (int64_t s = static_cast<int64_t>(blockIdx.x) * kR1Threads + threadIdx.x; s <= n;
       s += static_cast<int64_t>(gridDim.x) * kR1Threads) {
    const long long v = c0 + pref[s] + sums[s / kR1Scan];
    if (v > c) {
      c = v;
      st = s;
    }
  }
  long long oc, os;
  if (r1_best_reduce(c, st, bv, bs, counter, &oc, &os)) {
    *best_state = os == 0x7fffffffffffffffll ? 0 : os;
    *best_cut = oc;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

constexpr int kR1BestBlocks = 152 * 4;

struct R1Layout {
  int64_t n, npad, nscan_blocks, nscan_blocks_diff, nsort_blocks;
  size_t off_key, off_idx, off_code0, off_code_rank, off_d, off_sums, off_base, off_diff, off_dsums, off_counts,
      off_best, off_total, off_s0, off_cut0, off_state, off_state2, off_counter, total;
};

R1Layout r1_layout(int64_t n) {
  R1Layout l;
  l.n = n;
  l.npad = n;
  if (n <= kR1Bitonic) {
    l.npad = kR1Local;
    while (l.npad < n) l.npad <<= 1;
  }
  l.nscan_blocks = ceil_div(n, kR1Scan);
  l.nscan_blocks_diff = ceil_div(n + 1, kR1Scan);
  l.nsort_blocks = ceil_div(n, kR1Tile);
  size_t cur = 0;
  auto take = [&](size_t b) {
    size_t o = cur;
    cur = align_up(cur + b, 256);
    return o;
  };
  l.off_key = take(static_cast<size_t>(l.npad) * 8);
  l.off_idx = take(static_cast<size_t>(l.npad) * 4);
  l.off_code0 = take(static_cast<size_t>(n));
  l.off_code_rank = take(static_cast<size_t>(n) * 8);
  // the prefixes; while sorting, the other half of the (key, index) pairs
  l.off_d = take(static_cast<size_t>(n) * 16);
  l.off_sums = take(static_cast<size_t>(l.nscan_blocks) * 16);
  l.off_base = take(static_cast<size_t>(kR1BaseBlocks) * 16);
  l.off_diff = take(static_cast<size_t>(n + 2) * 8);
  l.off_dsums = take(static_cast<size_t>(l.nscan_blocks_diff) * 8);
  l.off_counts = take(static_cast<size_t>(l.nsort_blocks) * kR1Digits * 4);
  l.off_best = take(static_cast<size_t>(kR1BestBlocks) * 16);
  l.off_total = take(kR1Digits * 4);
  l.off_s0 = take(16);
  l.off_cut0 = take(8);
  l.off_state = take(8);
  l.off_state2 = take(8);
  l.off_counter = take(4);
  l.total = cur;
  return l;
}

}  // namespace

// two-eigenvector complex rounding vector (App. "Two-Eigenvector Complex
// Rounding", Eq. 12): q_i = u_1(i) + i u_2(i) from the real eigenvectors of
// a real symmetric Q, u_j = V_j / sqrt(lambda_j) (a column with
// lambda_j <= 0 contributes 0)
__global__ void r1_pair_kernel(const double2* __restrict__ V, int64_t n, int r, const double* __restrict__ lambda,
                               double2* __restrict__ q) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double l0 = lambda[0], l1 = lambda[1];
  const double s0 = l0 > 0.0 ? 1.0 / sqrt(l0) : 0.0, s1 = l1 > 0.0 ? 1.0 / sqrt(l1) : 0.0;
  q[i] = make_double2(V[i * r].x * s0, V[i * r + 1].x * s1);
}

int launch_two_eigvec_q(const double2* V, int64_t n, int r, const double* lambda, double2* q, cudaStream_t st) {
  r1_pair_kernel<<<static_cast<unsigned>(ceil_div(n, kR1Threads)), kR1Threads, 0, st>>>(V, n, r, lambda, q);
  count_launch();
  return cuda_check(cudaGetLastError(), "r1_pair_kernel");
}

size_t rank1_workspace_bytes(int64_t n) { return r1_layout(n).total; }

int launch_rank1(const double2* q, int64_t n, int K, uint8_t* z_out, double* f_out, const int32_t* rowptr,
                 const int32_t* colidx, int64_t nnz, int64_t* cut_out, uint8_t* zcut_out, void* ws, int32_t* status,
                 cudaStream_t st) {
  const R1Layout L = r1_layout(n);
  uint8_t* w = static_cast<uint8_t*>(ws);
  uint64_t* key = reinterpret_cast<uint64_t*>(w + L.off_key);
  uint32_t* idx = reinterpret_cast<uint32_t*>(w + L.off_idx);
  uint8_t* code0 = w + L.off_code0;
  uint2* code_rank = reinterpret_cast<uint2*>(w + L.off_code_rank);
  double2* d = reinterpret_cast<double2*>(w + L.off_d);
  uint64_t* key2 = reinterpret_cast<uint64_t*>(w + L.off_d);
  uint32_t* idx2 = reinterpret_cast<uint32_t*>(key2 + n);
  double2* sums = reinterpret_cast<double2*>(w + L.off_sums);
  double2* base = reinterpret_cast<double2*>(w + L.off_base);
  long long* diff = reinterpret_cast<long long*>(w + L.off_diff);
  long long* dsums = reinterpret_cast<long long*>(w + L.off_dsums);
  uint32_t* counts = reinterpret_cast<uint32_t*>(w + L.off_counts);
  uint32_t* total = reinterpret_cast<uint32_t*>(w + L.off_total);
  long long* bv = reinterpret_cast<long long*>(w + L.off_best);
  long long* bs = bv + kR1BestBlocks;
  double2* s0 = reinterpret_cast<double2*>(w + L.off_s0);
  unsigned long long* cut0 = reinterpret_cast<unsigned long long*>(w + L.off_cut0);
  int64_t* state = reinterpret_cast<int64_t*>(w + L.off_state);
  int64_t* state2 = reinterpret_cast<int64_t*>(w + L.off_state2);
  unsigned* counter = reinterpret_cast<unsigned*>(w + L.off_counter);
  R1Tables tb;
  Alphabet a = make_alphabet(K);
  for (int k = 0; k < kMaxK; ++k) {
    tb.zr[k] = k < K ? a.zr64[k] : 0.0;
    tb.zi[k] = k < K ? a.zi64[k] : 0.0;
  }
  int e = cuda_check(cudaMemsetAsync(counter, 0, sizeof(unsigned), st), "memset counter");
  if (e) return e;
  const int nbase = static_cast<int>(std::min<int64_t>(kR1BaseBlocks, ceil_div(L.npad, kR1Threads)));
  r1_prep_kernel<<<nbase, kR1Threads, 0, st>>>(q, n, L.npad, K, tb, key, idx, code0, base, counter, s0, status);
  count_launch();
  if (n <= kR1Bitonic) {
    const int npad = static_cast<int>(L.npad);
    const unsigned lb = static_cast<unsigned>(npad / kR1Local);
    r1_sort_local<<<lb, kR1Local / 2, 0, st>>>(key, idx, 2, kR1Local);
    count_launch();
    for (int k = 2 * kR1Local; k <= npad; k <<= 1) {
      for (int j = k >> 1; j >= kR1Local; j >>= 1) {
        r1_sort_global<<<static_cast<unsigned>(ceil_div(npad / 2, kR1Threads)), kR1Threads, 0, st>>>(key, idx, npad, k, j);
        count_launch();
      }
      r1_sort_local<<<lb, kR1Local / 2, 0, st>>>(key, idx, k, k);
      count_launch();
    }
  } else {
    if ((e = cuda_check(cudaFuncSetAttribute(r1_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kR1SortSmem),
                        "scatter shared memory")))
      return e;
    const unsigned sb = static_cast<unsigned>(L.nsort_blocks);
    uint64_t *ka = key, *kb = key2;
    uint32_t *ia = idx, *ib = idx2;
    for (int shift = 0; shift < 64; shift += 8) {  // an even number of passes: the result is in key, idx
      r1_hist_kernel<<<sb, kR1SortThreads, 0, st>>>(ka, n, shift, counts);
      r1_offsets_kernel<<<kR1Digits, kR1SortThreads, 0, st>>>(counts, L.nsort_blocks, total);
      r1_scatter_kernel<<<sb, kR1SortThreads, kR1SortSmem, st>>>(ka, ia, n, shift, counts, total, kb, ib);
      std::swap(ka, kb);
      std::swap(ia, ib);
      count_launch(3);
    }
  }
  r1_delta_scan_kernel<<<static_cast<unsigned>(L.nscan_blocks), kR1Threads, 0, st>>>(q, n, K, idx, code0, tb, d,
                                                                                     code_rank, sums, counter);
  const unsigned bb = static_cast<unsigned>(std::min<int64_t>(kR1BestBlocks, ceil_div(n, kR1Threads)));
  r1_best_kernel<<<bb, kR1Threads, 0, st>>>(d, n, sums, s0, bv, bs, counter, state, f_out);
  r1_codes_kernel<<<static_cast<unsigned>(ceil_div(n, 256)), 256, 0, st>>>(code_rank, n, K, state, z_out);
  count_launch(3);
  if (rowptr) {
    if ((e = cuda_check(cudaMemsetAsync(diff, 0, 8, st), "memset diff"))) return e;
    if ((e = cuda_check(cudaMemsetAsync(cut0, 0, 8, st), "memset cut0"))) return e;
    const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(n, kR1Threads), 152 * 8));
    r1_edge_kernel<<<blocks, kR1Threads, 0, st>>>(rowptr, colidx, n, nnz, K, code_rank, diff, cut0);
    r1_scan_kernel<<<static_cast<unsigned>(L.nscan_blocks_diff), kR1Threads, 0, st>>>(diff, n + 1, dsums, counter);
    const unsigned cb = static_cast<unsigned>(std::min<int64_t>(kR1BestBlocks, ceil_div(n + 1, kR1Threads)));
    r1_best_cut_kernel<<<cb, kR1Threads, 0, st>>>(diff, n, dsums, cut0, bv, bs, counter, state2, cut_out);
    r1_codes_kernel<<<static_cast<unsigned>(ceil_div(n, 256)), 256, 0, st>>>(code_rank, n, K, state2, zcut_out);
    count_launch(4);
  }
  return cuda_check(cudaGetLastError(), "rank-1 sweep kernels");
}

}  // namespace lrq
