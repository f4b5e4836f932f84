// k_batched.cu -- many independent instances of uneven n, r and K scored in
// one persistent launch (the sampling method of Sec. 4.2 applied per
// instance), with per-class tile shapes picked by the library's autotuner.
//
// Work decomposition: an item is (problem p, a tile of T consecutive
// candidates); it scores those T directions against all n_p coordinates, so
// items are independent and need no cross-item reduction.  A block of 64
// threads holds T candidates (four per thread) x (256 / T) row groups, or of
// 256 threads where the items are few (one per thread, b_slots_per_thread); the
// row groups split the coordinates of each shared-memory stage and are combined
// in FP64 at the end of the item.  Items are sorted by cost (n_p T) longest first
// and pulled by the persistent blocks from an atomic counter.
//
// Per problem the launch sequence is: input checks, direction sampling
// (Philox, when the caller passes no directions), the persistent scoring
// kernel (FP32 projections, sector decision by boundary signs, FP32 sums
// flushed to FP64 per stage), then one block per problem selects the top-m
// keys and re-scores them in FP64 (decision and sums in FP64), and keeps
// the best (ties to the smaller candidate index).
//
// Exact sub-batch: a problem given with S = 0 is solved exactly by vertex
// enumeration (Sec. 3, Algorithm 2) in the same persistent launch.  Its
// index sets, levels d = r..1 in turn, are cut into chunks of kBEnumChunk
// consecutive ranks; a chunk is one work item (FP64 null vectors and
// candidate scores, as in the standalone solver), whose best candidate goes
// to the problem's slot for that chunk, and the selection step reduces the
// chunks in the solver's deterministic order.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "batched_score.cuh"
#include "enum_device.cuh"
#include "gauss_df32.cuh"
#include "lrq_device.cuh"
#include "lrq_internal.h"
#include "score_f32x2.cuh"

namespace lrq {

constexpr int kBSelThreads = 256; // selection kernel
constexpr int kBMaxS = 8192;      // candidates per problem
constexpr int kBMaxTopM = 16;
constexpr int kBTiles[3] = {64, 128, 256};
constexpr double kBEnumBudget = 1e10;                            // r n^(2r+1) of one exact problem

// decision tables for K = 0..64 (entries below 2 unused), filled once per device
static __device__ BTable g_btab[kMaxK + 1];
// the exact solver's tables for K = 2..8
static __device__ EnumTables g_etab[kMaxTcK + 1];

// ---------------------------------------------------------------------------
// direction sampling and input checks
// ---------------------------------------------------------------------------
// Double-float (gauss_df32.cuh): 512 instances of up to 8192 directions take 0.34
// ms, 2.7 in FP64.
__global__ void __launch_bounds__(kSphereThreads) batched_sample_kernel(const BProb* __restrict__ probs,
                                                                        const int64_t* __restrict__ epoch) {
  const BProb& pb = probs[blockIdx.y];
  const int64_t s0 = static_cast<int64_t>(blockIdx.x) * sphere_per_block(pb.r);
  if (!pb.gen || s0 >= pb.S) return;
  sphere_block(pb.seed + static_cast<uint64_t>(*epoch), s0, pb.S, pb.r, const_cast<float2*>(pb.C));
}

__global__ void batched_check_kernel(const BProb* __restrict__ probs, int32_t* status) {
  const BProb pb = probs[blockIdx.y];
  const int64_t nv = 2 * pb.n * pb.r, nc = pb.gen ? 0 : 2 * static_cast<int64_t>(pb.S) * pb.r;
  const float* v = reinterpret_cast<const float*>(pb.V);
  const float* c = reinterpret_cast<const float*>(pb.C);
  bool bad = false;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < nv + nc;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x)
    bad |= !isfinite(t < nv ? v[t] : c[t - nv]);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) dev_fail(status, LRQ_EINVAL);
}

// ---------------------------------------------------------------------------
// per problem: top-m keys, FP64 re-scoring, winner
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t b_block_max(uint64_t v, uint64_t* red) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    const uint64_t o = __shfl_xor_sync(0xffffffffu, v, m);
    v = o > v ? o : v;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  uint64_t b = red[0];
  for (int k = 1; k < kBSelThreads / 32; ++k) b = red[k] > b ? red[k] : b;
  return b;
}

template <int R>
__device__ double b_rescore(const BProb& pb, int s, double* red) {
  double cr[R], ci[R], acc[2 * R];
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const float2 c = pb.C[static_cast<int64_t>(s) * R + j];
    cr[j] = c.x;
    ci[j] = c.y;
    acc[2 * j] = acc[2 * j + 1] = 0.0;
  }
  const BTable& tb = g_btab[pb.K];
  for (int64_t i = threadIdx.x; i < pb.n; i += kBSelThreads) {
    double vr[R], vi[R], x = 0.0, y = 0.0;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const float2 v = pb.V[i * R + j];
      vr[j] = v.x;
      vi[j] = v.y;
      x = fma(vr[j], cr[j], fma(-vi[j], ci[j], x));
      y = fma(vr[j], ci[j], fma(vi[j], cr[j], y));
    }
    const int k = decide_fp64(x, y, pb.K, tb.bcos64, tb.bsin64);
    const double zr = tb.zr64[k], zi = tb.zi64[k];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      acc[2 * j] = fma(vr[j], zr, fma(vi[j], zi, acc[2 * j]));
      acc[2 * j + 1] = fma(vr[j], zi, fma(-vi[j], zr, acc[2 * j + 1]));
    }
  }
  double f = 0.0;
#pragma unroll
  for (int j = 0; j < 2 * R; ++j) {
    double v = acc[j];
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int k = 0; k < kBSelThreads / 32; ++k) t += red[k];
    f += t * t;
  }
  return f;
}

// Exact problem: the best of its chunk results, in the solver's order.
__device__ void b_select_exact(const BProb& pb, const EnumBest* __restrict__ ebest, double* best_f, int64_t* best_idx,
                               int32_t* status) {
  __shared__ EnumBest sb[kBSelThreads];
  EnumBest best;
  best.f = -1.0;
  best.level = 0;
  best.sign = 1;
  best.rank = 0;
  best.choice = 0;
  for (int c = threadIdx.x; c < pb.nchunks; c += kBSelThreads)
    if (enum_better(ebest[pb.eb_off + c], best)) best = ebest[pb.eb_off + c];
  sb[threadIdx.x] = best;
  __syncthreads();
  for (int h = kBSelThreads / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h && enum_better(sb[threadIdx.x + h], sb[threadIdx.x])) sb[threadIdx.x] = sb[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    // no index set of full rank at any level (V's first column is zero)
    if (sb[0].f < 0.0) dev_fail(status, LRQ_EUNSUPPORTED);
    best_f[blockIdx.x] = sb[0].f;
    best_idx[blockIdx.x] = -1;
  }
}

// V^H z of a candidate as unit sums, K in {2, 3, 4, 6, 8}: omega^k = i^q (a + b
// tau) with a, b in {-1, 0, 1} and q in {0, 1}, so that conj(V_i) omega^k adds
// conj(V_i), turned or not, to A, B or both, V^H z = A + tau B, without products.
// The sums are exact three-word FP32 (two-sums twice).  The decision is certified
// in FP32 as in the re-scoring kernel, else taken in FP64.
constexpr int kBWarps = kBSelThreads / 32;
__device__ __forceinline__ bool b_unit_alphabet(int K) { return K == 2 || K == 3 || K == 4 || K == 6 || K == 8; }
__device__ __forceinline__ float4 b_unit_entry(int K, int k) {  // {a, b, turned, -}
  if (K == 8) {
    const float m = k < 4 ? 1.f : -1.f;
    return make_float4(k & 1 ? 0.f : m, k & 1 ? m : 0.f, static_cast<float>((k >> 1) & 1), 0.f);
  }
  if (K == 2 || K == 4) {
    const int q = K == 2 ? 2 * k : k;
    return make_float4(q < 2 ? 1.f : -1.f, 0.f, static_cast<float>(q & 1), 0.f);
  }
  const int t = K == 3 ? 2 * k : k;  // powers of tau = exp(i pi / 3): 1, tau, tau - 1, -1, -tau, 1 - tau
  const float a = t == 0 || t == 5 ? 1.f : (t == 2 || t == 3 ? -1.f : 0.f);
  const float b = t == 1 || t == 2 ? 1.f : (t == 4 || t == 5 ? -1.f : 0.f);
  return make_float4(a, b, 0.f, 0.f);
}

// The 2 r sums of candidate s over the rows of warp w of nw, to out; r <= R.
template <int R>
__device__ void b_unit_sums(const BProb& pb, int s, int w, int nw, const float4* __restrict__ unit, double* out) {
  const BTable& tb = g_btab[pb.K];
  const int K = pb.K, BK = K % 2 == 0 ? K / 2 : K, lane = threadIdx.x & 31;
  float cr[R], ci[R], mx = 0.f;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const float2 c = j < pb.r ? pb.C[static_cast<int64_t>(s) * pb.r + j] : make_float2(0.f, 0.f);
    cr[j] = c.x;
    ci[j] = c.y;
    mx = fmaxf(mx, fabsf(c.x) + fabsf(c.y));
  }
  // the error of an FP32 boundary projection is below cb sum_j |V_ij|_1 + 2^-140
  // where nothing overflows (fp32_row_bound, fp32_dir_bound)
  const float cb = fp32_dir_bound(mx, R);
  f32x2 hi[2][R], lo[2][R], l3[2][R];
#pragma unroll
  for (int g = 0; g < 2; ++g)
#pragma unroll
    for (int j = 0; j < R; ++j) hi[g][j] = lo[g][j] = l3[g][j] = 0;
  for (int64_t i = w * 32 + lane; i < pb.n; i += nw * 32) {
    float2 v[R];
    float x = 0.f, y = 0.f, ab = 0.f;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      v[j] = j < pb.r ? pb.V[i * pb.r + j] : make_float2(0.f, 0.f);
      ab += fabsf(v[j].x) + fabsf(v[j].y);
      x = fmaf(v[j].x, cr[j], x);
      x = fmaf(-v[j].y, ci[j], x);
      y = fmaf(v[j].x, ci[j], y);
      y = fmaf(v[j].y, cr[j], y);
    }
    uint32_t sb = 0;
    float pmin = INFINITY;
    for (int m = 0; m < BK; ++m) {
      const float p = fmaf(y, tb.bcos[m], -x * tb.bsin[m]);
      sb |= (p > 0.0f ? 1u : 0u) << m;
      pmin = fminf(pmin, fabsf(p));
    }
    int k;
    if (pmin > fp32_proj_bound(fp32_row_bound(ab), cb)) {
      if (K % 2 == 0) {
        const int c = __popc(sb);
        k = (sb & 1u) ? c : (c == 0 ? 0 : K - c);
      } else {
        const uint32_t t = sb & ~(sb >> 1) & ((1u << (K - 1)) - 1u);
        k = t ? __ffs(t) : 0;
      }
    } else {
      double xd = 0.0, yd = 0.0;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const double vr = v[j].x, vi = v[j].y, dr = cr[j], di = ci[j];
        xd = fma(vr, dr, fma(-vi, di, xd));
        yd = fma(vr, di, fma(vi, dr, yd));
      }
      k = decide_fp64(xd, yd, K, tb.bcos64, tb.bsin64);
    }
    const float4 u = unit[k];
    const f32x2 ua = pack2(u.x, u.x), ub = pack2(u.y, u.y);
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const f32x2 vv = u.z != 0.f ? pack2(v[j].y, v[j].x) : pack2(v[j].x, -v[j].y);  // i conj(V_ij) or conj(V_ij)
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        const f32x2 e = add_unit(hi[g][j], vv, g ? ub : ua);
        l3[g][j] = add2(l3[g][j], add_unit(lo[g][j], e, pack2(1.f, 1.f)));
      }
    }
  }
  // the lanes' sums in FP64; 16 values at a time, halved at every step
  const double tr = K == 8 ? 0.70710678118654752440 : 0.5;
  const double ti = K == 8 ? 0.70710678118654752440 : 0.86602540378443864676;
  const bool both = K != 2 && K != 4;
  double val[16];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    val[2 * j] = val[2 * j + 1] = 0.0;
    if (j < R) {
      double a[2][2];
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        a[g][0] = a[g][1] = 0.0;
        if (g == 0 || both) {
          float h0, h1, m0, m1, t0, t1;
          unpack2(hi[g][j < R ? j : 0], h0, h1);
          unpack2(lo[g][j < R ? j : 0], m0, m1);
          unpack2(l3[g][j < R ? j : 0], t0, t1);
          a[g][0] = static_cast<double>(h0) + (static_cast<double>(m0) + static_cast<double>(t0));
          a[g][1] = static_cast<double>(h1) + (static_cast<double>(m1) + static_cast<double>(t1));
        }
      }
      val[2 * j] = a[0][0];
      val[2 * j + 1] = a[0][1];
      if (both) {
        val[2 * j] += tr * a[1][0] - ti * a[1][1];
        val[2 * j + 1] += tr * a[1][1] + ti * a[1][0];
      }
    }
  }
#pragma unroll
  for (int k = 8, m = 16; k > 0; k >>= 1, m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int q = 0; q < k; ++q) {
      const double give = up ? val[q] : val[k + q], keep = up ? val[k + q] : val[q];
      val[q] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
  }
  val[0] += __shfl_xor_sync(0xffffffffu, val[0], 1);
  if ((lane & 1) == 0) out[lane >> 1] = val[0];
}

// One block per problem.  The keys are read once, into registers; the selected
// candidates are re-scored side by side, the warps shared out among them (unit
// alphabets), or one after the other in FP64.  512 instances, four candidates
// each: 889 us with every candidate in FP64 by the whole block, now 303.
__global__ void __launch_bounds__(kBSelThreads) batched_select_kernel(const BProb* __restrict__ probs,
                                                                   const uint64_t* __restrict__ keys, int top_m,
                                                                   const EnumBest* __restrict__ ebest,
                                                                   double* __restrict__ best_f,
                                                                   int64_t* __restrict__ best_idx,
                                                                   int64_t* __restrict__ epoch,
                                                                   int32_t* __restrict__ status) {
  __shared__ uint64_t redk[kBSelThreads / 32];
  __shared__ double redd[kBSelThreads / 32];
  const BProb pb = probs[blockIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0) *epoch += 1;  // the next call draws fresh directions
  if (pb.exact) {
    b_select_exact(pb, ebest, best_f, best_idx, status);
    return;
  }
  __shared__ double part[kBWarps][16];
  __shared__ float4 unit[8];
  __shared__ int chosen[kBMaxTopM];
  __shared__ double fq[kBMaxTopM];
  const uint64_t* kp = keys + pb.key_off;
  const int m = min(top_m, pb.S);
  const bool fast = b_unit_alphabet(pb.K);
  if (fast && threadIdx.x < pb.K) unit[threadIdx.x] = b_unit_entry(pb.K, threadIdx.x);
  constexpr int kKeys = kBMaxS / kBSelThreads;
  uint64_t key[kKeys];
#pragma unroll
  for (int q = 0; q < kKeys; ++q) {
    const int s = threadIdx.x + q * kBSelThreads;
    key[q] = s < pb.S ? kp[s] : 0ull;
  }
  int got = 0;
  uint64_t prev = ~0ull;
  for (; got < m; ++got) {
    uint64_t v = 0;
#pragma unroll
    for (int q = 0; q < kKeys; ++q)
      if (key[q] < prev && key[q] > v) v = key[q];
    const uint64_t kmax = b_block_max(v, redk);
    prev = kmax;
    const int s = static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(kmax & 0xFFFFFFFFull));
    if (kmax == 0 || s < 0 || s >= pb.S) break;  // no key left (block-uniform)
    if (threadIdx.x == 0) chosen[got] = s;
  }
  __syncthreads();
  double bf = -1.0;
  int bs = 0;
  bool all64 = !fast;
  if (fast) {
    // warps per candidate; candidates q0 .. q0 + kBWarps / per - 1 at a time
    const int per = got >= kBWarps ? 1 : (got >= 5 ? 1 : (got >= 3 ? 2 : (got == 2 ? 4 : 8)));
    const int warp = threadIdx.x >> 5, at_once = kBWarps / per;
    for (int q0 = 0; q0 < got; q0 += at_once) {
      const int q = q0 + warp / per;
      if (q < got) {
        const int s = chosen[q];
        if (pb.r <= 2)
          b_unit_sums<2>(pb, s, warp % per, per, unit, part[warp]);
        else if (pb.r <= 4)
          b_unit_sums<4>(pb, s, warp % per, per, unit, part[warp]);
        else
          b_unit_sums<8>(pb, s, warp % per, per, unit, part[warp]);
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int c = 0; c < at_once && q0 + c < got; ++c) {
          double f = 0.0;
          for (int j = 0; j < 2 * pb.r; ++j) {
            double v = part[c * per][j];
            for (int w = 1; w < per; ++w) v += part[c * per + w][j];
            f += v * v;
          }
          fq[q0 + c] = f;
        }
      }
      __syncthreads();
    }
    for (int q = 0; q < got; ++q) {
      bf = fmax(bf, fq[q]);
      all64 |= !isfinite(fq[q]);  // FP32 sums of entries around 10^38 overflow
    }
  }
  // the best in FP64's own order: directions whose assignments are turns of one
  // another have the same f, which only rounding tells apart, so values this
  // close are taken again in FP64 as for the other alphabets
  const double near = all64 ? -1.0 : bf * (1.0 - 1e-10);
  int close = 0;
  for (int q = 0; q < got; ++q) {
    if (all64 || fq[q] >= near) {
      ++close;
      bs = chosen[q];
    }
  }
  if (all64 || close > 1) {
    bf = -1.0;
    for (int q = 0; q < got; ++q) {
      if (!all64 && !(fq[q] >= near)) continue;
      const int s = chosen[q];
      double f;
      switch (pb.r) {
        case 1: f = b_rescore<1>(pb, s, redd); break;
        case 2: f = b_rescore<2>(pb, s, redd); break;
        case 3: f = b_rescore<3>(pb, s, redd); break;
        case 4: f = b_rescore<4>(pb, s, redd); break;
        case 5: f = b_rescore<5>(pb, s, redd); break;
        case 6: f = b_rescore<6>(pb, s, redd); break;
        case 7: f = b_rescore<7>(pb, s, redd); break;
        default: f = b_rescore<8>(pb, s, redd); break;
      }
      if (f > bf || (f == bf && s < bs)) {
        bf = f;
        bs = s;
      }
    }
  }
  if (threadIdx.x == 0) {
    if (bf < 0.0) dev_fail(status, LRQ_EINVAL);
    best_f[blockIdx.x] = bf;
    best_idx[blockIdx.x] = bs;
  }
}

// ---------------------------------------------------------------------------
// host side: plan, workspace, launch sequence, autotuner, graph
// ---------------------------------------------------------------------------
struct lrq_batched_plan_impl {
  std::vector<lrq_problem> probs;
  std::vector<int> tile;
  int top_m = 0;
  int device = 0;
  int grid_wide = 0, grid = 0;  // resident blocks of batched_score_kernel<1> and <4>
  int64_t nkeys = 0, ncgen = 0;
  size_t off_probs = 0, off_items = 0, off_counter = 0, off_epoch = 0, off_keys = 0, off_C = 0, off_ebest = 0,
         total = 0;
  int64_t nebest = 0;
  int nitems = 0;
  int per_thread = 4;     // slots per thread of the scoring kernel
  const BTable* btab = nullptr;  // the device's decision tables, from prepare on
  const EnumTables* etab = nullptr;
  int sample_blocks = 0;  // of the problem with most directions to draw
  bool prepared = false;
  const void* prepared_ws = nullptr;
};

namespace {

std::mutex g_btab_mu;
bool g_btab_ready[64] = {};
std::mutex g_tile_mu;
std::map<std::tuple<int, int, int, int>, int> g_tile_cache;  // (device, r, K, log2 n) -> tile

int n_bucket(int64_t n) {
  int b = 0;
  while ((int64_t(1) << (b + 1)) <= n) ++b;
  return b;
}

int ensure_tables(int dev) {
  std::lock_guard<std::mutex> lk(g_btab_mu);
  if (dev < 0 || dev >= 64) return fail(LRQ_EUNSUPPORTED, "device index above 63");
  if (g_btab_ready[dev]) return LRQ_OK;
  std::vector<BTable> t(kMaxK + 1);
  std::memset(t.data(), 0, t.size() * sizeof(BTable));
  for (int K = 2; K <= kMaxK; ++K) {
    Alphabet a = make_alphabet(K);
    for (int m = 0; m < 8; ++m) {
      t[K].bcos[m] = m < a.BK ? a.bcos[m] : 0.f;
      t[K].bsin[m] = m < a.BK ? a.bsin[m] : 0.f;
      t[K].bcos64[m] = m < a.BK ? a.bcos64[m] : 0.0;
      t[K].bsin64[m] = m < a.BK ? a.bsin64[m] : 0.0;
    }
    for (int k = 0; k < K; ++k) {
      t[K].zr[k] = a.zr[k];
      t[K].zi[k] = a.zi[k];
      t[K].zr64[k] = a.zr64[k];
      t[K].zi64[k] = a.zi64[k];
    }
  }
  int e = cuda_check(cudaMemcpyToSymbol(g_btab, t.data(), t.size() * sizeof(BTable)), "upload decision tables");
  if (e) return e;
  std::vector<EnumTables> et(kMaxTcK + 1);
  std::memset(et.data(), 0, et.size() * sizeof(EnumTables));
  for (int K = 2; K <= kMaxTcK; ++K) et[K] = make_enum_tables(K);
  if ((e = cuda_check(cudaMemcpyToSymbol(g_etab, et.data(), et.size() * sizeof(EnumTables)),
                      "upload enumeration tables")))
    return e;
  g_btab_ready[dev] = true;
  return LRQ_OK;
}

// Index sets of an exact problem's levels d = 1..r, and its work items.
void exact_levels(const lrq_problem& q, unsigned long long* lvl) {
  const int BK = (q.K % 2 == 0) ? q.K / 2 : q.K;
  for (int d = 1; d <= kEnumMaxD; ++d) lvl[d - 1] = d <= q.r ? binom(static_cast<int>(q.n) * BK, 2 * d - 1) : 0ull;
}

int64_t exact_chunks(const lrq_problem& q) {
  unsigned long long lvl[kEnumMaxD], total = 0;
  exact_levels(q, lvl);
  for (int d = 0; d < kEnumMaxD; ++d) total += lvl[d];
  return static_cast<int64_t>((total + kBEnumChunk - 1) / kBEnumChunk);
}

void layout(lrq_batched_plan_impl* pl) {
  size_t cur = 0;
  auto take = [&](size_t bytes) {
    size_t o = cur;
    cur = align_up(cur + bytes, 256);
    return o;
  };
  const int P = static_cast<int>(pl->probs.size());
  int64_t nitems = 0;
  pl->nkeys = 0;
  pl->ncgen = 0;
  pl->nebest = 0;
  for (const lrq_problem& q : pl->probs) {
    if (q.S == 0) {  // exact
      const int64_t ch = exact_chunks(q);
      nitems += ch;
      pl->nebest += ch;
      continue;
    }
    nitems += ceil_div(q.S, kBTiles[0]);  // room for the smallest tile
    pl->nkeys += q.S;
    if (!q.C) {
      pl->ncgen += q.S * q.r;
      pl->sample_blocks = std::max(pl->sample_blocks, static_cast<int>(ceil_div(q.S, sphere_per_block(q.r))));
    }
  }
  pl->off_probs = take(static_cast<size_t>(P) * sizeof(BProb));
  pl->off_items = take(static_cast<size_t>(nitems) * sizeof(BItem));
  pl->off_counter = take(sizeof(int));
  pl->off_epoch = take(sizeof(int64_t));
  pl->off_keys = take(static_cast<size_t>(pl->nkeys) * sizeof(uint64_t));
  pl->off_C = take(static_cast<size_t>(pl->ncgen) * sizeof(float2));
  pl->off_ebest = take(static_cast<size_t>(pl->nebest) * sizeof(EnumBest));
  pl->total = cur;
}

// Slots per thread of the scoring kernel: four (fewest instructions an
// evaluation) once the items' cost fills the resident blocks a good deal longer
// than the longest item takes in one of them; below that the longest items, or
// the last of them, are the launch's time, and a block of 256 threads takes
// about half of it.  Measured with one / four slots a thread, by total over
// longest item (four slots: 912 resident blocks): 26 126 / 176 us, 163 971 /
// 2260, 330 179 / 250, 651 1849 / 2313, 892 773 / 730, 934 814 / 815, 1024 equal
// items 364 / 352 (r = 4, K = 3) and 638 / 800 (r = 8), 1216 3858 / 3428, 4863
// 14308 / 11794.
// One slot also where most of the work is of a kind that gains nothing from four:
// exact items (FP64 out of local memory; a unit of their cost takes about 24 times
// a scoring item's; 64 with n = 24: 31.4 / 40.7 ms), K > 8 (the angle; 200 of
// K = 11: 3494 / 3838 us) and K = 5, 6, 7 (b_dispatch_k; 200 of K = 5: 1965 /
// 2501 us).
// Either form adds the same numbers in the same order.
int b_slots_per_thread(const lrq_batched_plan_impl* pl, double scoring, double other, double longest) {
  return other > scoring || scoring + other < 1.25 * longest * pl->grid ? 1 : 4;
}

// Device descriptors and the item list for the problems in `subset` (all
// when empty), with the plan's current tiles.
int upload(lrq_batched_plan_impl* pl, uint8_t* ws, const std::vector<int>& subset, cudaStream_t st, int* nitems_out,
           int* per_thread_out) {
  const int P = static_cast<int>(pl->probs.size());
  std::vector<BProb> hp(P);
  int64_t key_off = 0, c_off = 0, eb_off = 0;
  float2* Cgen = reinterpret_cast<float2*>(ws + pl->off_C);
  for (int p = 0; p < P; ++p) {
    const lrq_problem& q = pl->probs[p];
    BProb b;
    std::memset(&b, 0, sizeof(b));
    b.V = static_cast<const float2*>(q.V);
    if (q.S == 0) {
      b.exact = 1;
      b.n = q.n;
      b.r = q.r;
      b.K = q.K;
      exact_levels(q, b.lvl_total);
      b.nchunks = static_cast<int>(exact_chunks(q));
      b.eb_off = eb_off;
      eb_off += b.nchunks;
      hp[p] = b;
      continue;
    }
    b.gen = q.C ? 0 : 1;
    b.C = q.C ? static_cast<const float2*>(q.C) : Cgen + c_off;
    if (!q.C) c_off += q.S * q.r;
    b.n = q.n;
    b.r = q.r;
    b.K = q.K;
    b.S = static_cast<int>(q.S);
    b.tile = pl->tile[p];
    b.seed = q.seed;
    b.key_off = key_off;
    key_off += q.S;
    hp[p] = b;
  }
  std::vector<int> which = subset;
  if (which.empty())
    for (int p = 0; p < P; ++p) which.push_back(p);
  std::vector<BItem> items;
  for (int p : which) {
    if (hp[p].exact) {
      for (int c = 0; c < hp[p].nchunks; ++c) items.push_back(BItem{p, c});
      continue;
    }
    for (int s0 = 0; s0 < hp[p].S; s0 += hp[p].tile) items.push_back(BItem{p, s0});
  }
  // longest first: cost ~ n_p * tile * (r_p + 1) FP32 lane operations for a
  // scoring item; an exact item's kBEnumChunk index sets each cost two
  // vertices of about n_p (4 d + 24) FP64 operations, weighted 32x
  auto cost = [&](const BItem& it) {
    const BProb& b = hp[it.p];
    if (b.exact) return static_cast<double>(b.n) * kBEnumChunk * 2.0 * (4.0 * b.r + 24.0) * 32.0 / kBSlots;
    return static_cast<double>(b.n) * b.tile * (b.r + 1);
  };
  std::stable_sort(items.begin(), items.end(), [&](const BItem& a, const BItem& b) { return cost(a) > cost(b); });
  int e = cuda_check(cudaMemcpyAsync(ws + pl->off_probs, hp.data(), hp.size() * sizeof(BProb),
                                     cudaMemcpyHostToDevice, st),
                     "upload problems");
  if (e) return e;
  if (!items.empty() &&
      (e = cuda_check(cudaMemcpyAsync(ws + pl->off_items, items.data(), items.size() * sizeof(BItem),
                                      cudaMemcpyHostToDevice, st),
                      "upload items")))
    return e;
  if ((e = cuda_check(cudaStreamSynchronize(st), "upload sync"))) return e;  // host vectors end here
  *nitems_out = static_cast<int>(items.size());
  double scoring = 0.0, other = 0.0;
  for (const BItem& it : items) {
    const BProb& b = hp[it.p];
    if (b.exact)
      other += 24.0 * cost(it);
    else
      (b.K <= 4 || b.K == 8 ? scoring : other) += cost(it);
  }
  *per_thread_out = b_slots_per_thread(pl, scoring, other, items.empty() ? 0.0 : cost(items[0]));
  return LRQ_OK;
}

int launch_sequence(const lrq_batched_plan_impl* pl, uint8_t* ws, int nitems, int per_thread, bool sample, bool select,
                    double* best_f, int64_t* best_idx, int32_t* status, cudaStream_t st) {
  const int P = static_cast<int>(pl->probs.size());
  const BProb* probs = reinterpret_cast<const BProb*>(ws + pl->off_probs);
  int64_t* epoch = reinterpret_cast<int64_t*>(ws + pl->off_epoch);
  int* counter = reinterpret_cast<int*>(ws + pl->off_counter);
  uint64_t* keys = reinterpret_cast<uint64_t*>(ws + pl->off_keys);
  if (sample) {
    batched_check_kernel<<<dim3(64, P), 256, 0, st>>>(probs, status);
    count_launch();
    if (pl->sample_blocks > 0) {
      batched_sample_kernel<<<dim3(pl->sample_blocks, P), kSphereThreads, 0, st>>>(probs, epoch);
      count_launch();
    }
  }
  int e = cuda_check(cudaMemsetAsync(counter, 0, sizeof(int), st), "reset item counter");
  if (e) return e;
  timing_start(st);
  EnumBest* ebest = reinterpret_cast<EnumBest*>(ws + pl->off_ebest);
  const BItem* items = reinterpret_cast<const BItem*>(ws + pl->off_items);
  if (per_thread == 1)
    launch_batched_score<1>(pl->grid_wide, st, probs, items, nitems, counter, pl->btab, pl->etab, keys, ebest, status);
  else
    launch_batched_score<4>(pl->grid, st, probs, items, nitems, counter, pl->btab, pl->etab, keys, ebest, status);
  timing_stop(st);
  count_launch();
  if (select) {
    batched_select_kernel<<<P, kBSelThreads, 0, st>>>(probs, keys, pl->top_m, ebest, best_f, best_idx, epoch, status);
    count_launch();
  }
  return cuda_check(cudaGetLastError(), "batched kernels");
}

std::mutex g_graph_mu;
std::map<void*, int> g_graph_launches;  // graph exec -> kernels per replay

}  // namespace

}  // namespace lrq

using namespace lrq;

struct lrq_batched_plan : lrq_batched_plan_impl {};

extern "C" {

int lrq_batched_plan_create(const lrq_problem* problems, int P, int top_m, lrq_batched_plan** plan_out) {
  if (!plan_out) return fail(LRQ_EINVAL, "plan_out is NULL");
  *plan_out = nullptr;
  if (!problems || P < 1) return fail(LRQ_EINVAL, "need at least one problem");
  if (P > 65535) return fail(LRQ_EUNSUPPORTED, "at most 65535 problems per plan");
  if (top_m < 1 || top_m > kBMaxTopM) return fail(LRQ_EINVAL, "top_m must be in [1, 16]");
  for (int p = 0; p < P; ++p) {
    const lrq_problem& q = problems[p];
    if (!q.V) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": V is NULL");
    if (q.n < 1 || q.n >= (int64_t(1) << 31)) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": bad n");
    if (q.r < 1 || q.r > kMaxRank) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": r not in [1, 8]");
    if (q.K < 2 || q.K > kMaxK) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": K not in [2, 64]");
    if (q.S == 0) {  // exact sub-batch
      if (q.C) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": exact (S = 0) takes no directions");
      int e = enumerate_check(q.n, q.r, q.K, kBEnumBudget);
      if (e) return fail(e, "problem " + std::to_string(p) + " (exact): " + lrq_last_error());
      if (exact_chunks(q) > (int64_t(1) << 24))
        return fail(LRQ_EUNSUPPORTED, "problem " + std::to_string(p) + ": too many index sets");
      continue;
    }
    if (q.S < 1 || q.S > kBMaxS) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": S not in [0, 8192]");
    if (top_m > q.S) return fail(LRQ_EINVAL, "problem " + std::to_string(p) + ": top_m > S");
  }
  int dev = 0;
  int e = cuda_check(cudaGetDevice(&dev), "cudaGetDevice");
  if (e) return e;
  lrq_batched_plan* pl = new lrq_batched_plan();
  pl->probs.assign(problems, problems + P);
  pl->top_m = top_m;
  pl->device = dev;
  pl->tile.resize(P);
  {
    std::lock_guard<std::mutex> lk(g_tile_mu);
    for (int p = 0; p < P; ++p) {
      auto it = g_tile_cache.find(std::make_tuple(dev, pl->probs[p].r, pl->probs[p].K, n_bucket(pl->probs[p].n)));
      pl->tile[p] = it != g_tile_cache.end() ? it->second : 128;
    }
  }
  int per_sm = 1, per_sm_wide = 1;
  if ((e = batched_blocks_per_sm<4>(&per_sm)) || (e = batched_blocks_per_sm<1>(&per_sm_wide))) {
    delete pl;
    return e;
  }
  pl->grid = std::max(1, per_sm) * num_sms_current();
  pl->grid_wide = std::max(1, per_sm_wide) * num_sms_current();
  layout(pl);
  *plan_out = pl;
  return LRQ_OK;
}

void lrq_batched_plan_destroy(lrq_batched_plan* plan) { delete plan; }

int lrq_batched_workspace_size(const lrq_batched_plan* plan, size_t* bytes) {
  if (!plan || !bytes) return fail(LRQ_EINVAL, "NULL argument");
  *bytes = plan->total;
  return LRQ_OK;
}

int lrq_batched_prepare(lrq_batched_plan* plan, void* ws, size_t ws_bytes, void* stream) {
  if (!plan) return fail(LRQ_EINVAL, "plan is NULL");
  if (!ws || reinterpret_cast<uintptr_t>(ws) % 256 != 0 || ws_bytes < plan->total)
    return fail(LRQ_EWORKSPACE, "workspace missing, misaligned or smaller than lrq_batched_workspace_size");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int e = ensure_tables(plan->device);
  if (e) return e;
  void *bt = nullptr, *et = nullptr;
  if ((e = cuda_check(cudaGetSymbolAddress(&bt, g_btab), "decision tables")) ||
      (e = cuda_check(cudaGetSymbolAddress(&et, g_etab), "enumeration tables")))
    return e;
  plan->btab = static_cast<const BTable*>(bt);
  plan->etab = static_cast<const EnumTables*>(et);
  uint8_t* w = static_cast<uint8_t*>(ws);
  if ((e = cuda_check(cudaMemsetAsync(w + plan->off_epoch, 0, sizeof(int64_t), st), "reset epoch"))) return e;
  if ((e = upload(plan, w, {}, st, &plan->nitems, &plan->per_thread))) return e;
  plan->prepared = true;
  plan->prepared_ws = ws;
  return LRQ_OK;
}

int lrq_sample_score_batched(const lrq_batched_plan* plan, void* ws, size_t ws_bytes, double* best_f_out,
                             int64_t* best_idx_out, int32_t* dev_status, void* stream) {
  if (!plan || !best_f_out || !best_idx_out || !dev_status) return fail(LRQ_EINVAL, "NULL pointer argument");
  if (!plan->prepared || plan->prepared_ws != ws || ws_bytes < plan->total)
    return fail(LRQ_EINVAL, "call lrq_batched_prepare with this workspace first");
  return launch_sequence(plan, static_cast<uint8_t*>(ws), plan->nitems, plan->per_thread, true, true, best_f_out, best_idx_out,
                         dev_status, static_cast<cudaStream_t>(stream));
}

int lrq_batched_autotune(lrq_batched_plan* plan, void* ws, size_t ws_bytes, int32_t* dev_status, void* stream) {
  if (!plan || !dev_status) return fail(LRQ_EINVAL, "NULL pointer argument");
  if (!plan->prepared || plan->prepared_ws != ws || ws_bytes < plan->total)
    return fail(LRQ_EINVAL, "call lrq_batched_prepare with this workspace first");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t* w = static_cast<uint8_t*>(ws);
  const int P = static_cast<int>(plan->probs.size());
  // directions once (the timed runs score them again and again)
  int e = launch_sequence(plan, w, 0, plan->per_thread, true, false, nullptr, nullptr, dev_status, st);
  if (e) return e;
  if ((e = cuda_check(cudaMemsetAsync(w + plan->off_epoch, 0, sizeof(int64_t), st), "reset epoch"))) return e;
  std::map<std::tuple<int, int, int>, std::vector<int>> classes;
  for (int p = 0; p < P; ++p)
    if (plan->probs[p].S > 0)
      classes[std::make_tuple(plan->probs[p].r, plan->probs[p].K, n_bucket(plan->probs[p].n))].push_back(p);
  cudaEvent_t t0, t1;
  if ((e = cuda_check(cudaEventCreate(&t0), "event"))) return e;
  if ((e = cuda_check(cudaEventCreate(&t1), "event"))) {
    cudaEventDestroy(t0);
    return e;
  }
  for (auto& kv : classes) {
    float best_ms = 0.f;
    int best_tile = 128;
    for (int ti = 0; ti < 3; ++ti) {
      for (int p : kv.second) plan->tile[p] = kBTiles[ti];
      int nit = 0, per_thread = 4;
      if ((e = upload(plan, w, kv.second, st, &nit, &per_thread))) break;
      float ms = 0.f;
      for (int rep = 0; rep < 3 && !e; ++rep) {
        cudaEventRecord(t0, st);
        e = launch_sequence(plan, w, nit, per_thread, false, false, nullptr, nullptr, dev_status, st);
        cudaEventRecord(t1, st);
        if (!e) e = cuda_check(cudaEventSynchronize(t1), "autotune sync");
        float x = 0.f;
        cudaEventElapsedTime(&x, t0, t1);
        ms = rep == 0 ? x : std::min(ms, x);
      }
      if (e) break;
      if (ti == 0 || ms < best_ms) {
        best_ms = ms;
        best_tile = kBTiles[ti];
      }
    }
    if (e) break;
    for (int p : kv.second) plan->tile[p] = best_tile;
    std::lock_guard<std::mutex> lk(g_tile_mu);
    g_tile_cache[std::make_tuple(plan->device, std::get<0>(kv.first), std::get<1>(kv.first),
                                 std::get<2>(kv.first))] = best_tile;
  }
  cudaEventDestroy(t0);
  cudaEventDestroy(t1);
  if (e) return e;
  return upload(plan, w, {}, st, &plan->nitems, &plan->per_thread);
}

int lrq_batched_tile(const lrq_batched_plan* plan, int p) {
  if (!plan || p < 0 || p >= static_cast<int>(plan->probs.size())) return -1;
  if (plan->probs[p].S == 0) return 0;  // exact: no candidate tile
  return plan->tile[p];
}

int lrq_batched_graph_create(const lrq_batched_plan* plan, void* ws, size_t ws_bytes, double* best_f_out,
                             int64_t* best_idx_out, int32_t* dev_status, void* stream, void** graph_exec_out) {
  if (!graph_exec_out) return fail(LRQ_EINVAL, "graph_exec_out is NULL");
  *graph_exec_out = nullptr;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (!st) return fail(LRQ_EINVAL, "graph capture needs a non-default stream");
  int e = cuda_check(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal), "begin capture");
  if (e) return e;
  const uint64_t before = lrq_kernel_launches();
  int e2 = lrq_sample_score_batched(plan, ws, ws_bytes, best_f_out, best_idx_out, dev_status, stream);
  const int nk = static_cast<int>(lrq_kernel_launches() - before);
  cudaGraph_t g = nullptr;
  e = cuda_check(cudaStreamEndCapture(st, &g), "end capture");
  if (e2 || e) {
    if (g) cudaGraphDestroy(g);
    return e2 ? e2 : e;
  }
  cudaGraphExec_t ex = nullptr;
  e = cuda_check(cudaGraphInstantiate(&ex, g, 0), "instantiate graph");
  cudaGraphDestroy(g);
  if (e) return e;
  // the capture counted its kernels; count them again on every replay instead
  count_launch(-nk);
  {
    std::lock_guard<std::mutex> lk(g_graph_mu);
    g_graph_launches[ex] = nk;
  }
  *graph_exec_out = ex;
  return LRQ_OK;
}

int lrq_graph_launch(void* graph_exec, void* stream) {
  if (!graph_exec) return fail(LRQ_EINVAL, "graph_exec is NULL");
  int nk = 0;
  {
    std::lock_guard<std::mutex> lk(g_graph_mu);
    auto it = g_graph_launches.find(graph_exec);
    if (it == g_graph_launches.end()) return fail(LRQ_EINVAL, "unknown graph");
    nk = it->second;
  }
  int e = cuda_check(cudaGraphLaunch(static_cast<cudaGraphExec_t>(graph_exec), static_cast<cudaStream_t>(stream)),
                     "cudaGraphLaunch");
  if (!e) count_launch(nk);
  return e;
}

int lrq_graph_destroy(void* graph_exec) {
  if (!graph_exec) return LRQ_OK;
  {
    std::lock_guard<std::mutex> lk(g_graph_mu);
    g_graph_launches.erase(graph_exec);
  }
  return cuda_check(cudaGraphExecDestroy(static_cast<cudaGraphExec_t>(graph_exec)), "cudaGraphExecDestroy");
}

}  // extern "C"
