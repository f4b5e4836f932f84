// k_score_fp32.cu -- direction sampler, input checks, column sums, CUDA-core
// FP32 candidate scoring and the per-candidate finalisation shared by both
// scoring modes.
//
// Scoring follows Sec. 4.2, Eq. 10: for direction c, w_i = V_i c, the decision
// rule of Sec. 3, Eq. 9 picks k_i, and f(c) = ||V^H z(c)||^2.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "gauss_df32.cuh"
#include "lrq_device.cuh"
#include "lrq_internal.h"
#include "score_f32x2.cuh"

namespace lrq {

// Uniform directions on the complex unit sphere (gauss_df32.cuh).  Bound:
// issue slots, about 250 instructions a component, and the candidates drawn again
// in FP64 (3.2 us without them).  S = 2^14, r = 4: 6.8 us, 26 in FP64 (two lanes an
// SM).
__global__ void __launch_bounds__(kSphereThreads) sample_directions_kernel(uint64_t seed, int64_t S, int r,
                                                                           float2* __restrict__ C) {
  sphere_block(seed, static_cast<int64_t>(blockIdx.x) * sphere_per_block(r), S, r, C);
}

int launch_sample_directions(uint64_t seed, int64_t S, int r, float2* C, cudaStream_t st) {
  if (S <= 0) return LRQ_OK;
  int64_t blocks = ceil_div(S, sphere_per_block(r));
  sample_directions_kernel<<<static_cast<unsigned>(blocks), kSphereThreads, 0, st>>>(seed, S, r, C);
  count_launch();
  return cuda_check(cudaGetLastError(), "sample_directions_kernel");
}

// ---------------------------------------------------------------------------
// Non-finite input check (the ABI reports LRQ_EINVAL through dev_status).
// ---------------------------------------------------------------------------
__global__ void check_finite_kernel(const float* __restrict__ x, int64_t count, int32_t* status) {
  int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  bool bad = false;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += stride)
    bad |= !isfinite(x[i]);
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) dev_fail(status, LRQ_EINVAL);
}

int launch_check_finite(const float* x, int64_t count, int32_t* status, cudaStream_t st) {
  if (count <= 0) return LRQ_OK;
  int blocks = static_cast<int>(std::min<int64_t>(ceil_div(count, 256), 4 * 152));
  check_finite_kernel<<<blocks, 256, 0, st>>>(x, count, status);
  count_launch();
  return cuda_check(cudaGetLastError(), "check_finite_kernel");
}

// ---------------------------------------------------------------------------
// One pass over V for the tensor-core mode: the finiteness check, each block's
// largest |component| and (sums) each block's part of T = sum_i conj(V_i) in
// FP64 (the class-0 base of the odd-K indicator form).  The packing kernel
// reduces the parts (in block order: deterministic).  Bound: FP64 (2r
// additions a row; the conversions from FP32 are integer operations, since a
// conversion instruction runs on the FP64 unit too).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double exact_double(float x) {
  const uint32_t b = __float_as_uint(x), e = (b >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) return static_cast<double>(x);  // zero, subnormal, infinite, NaN
  return __hiloint2double(static_cast<int>((b & 0x80000000u) | ((b & 0x7fffffffu) >> 3)) + (896 << 20),
                          static_cast<int>(b << 29));
}

// Sums 16 doubles over the warp, halving the values at every step (16 additions
// a lane instead of 80): lane l ends with the total of value l >> 1.
__device__ __forceinline__ double warp_sums16(double (&v)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 8, m = 16; k > 0; k >>= 1, m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int q = 0; q < k; ++q) {
      const double give = up ? v[q] : v[k + q], keep = up ? v[k + q] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

template <int R, bool SUMS>
__global__ void __launch_bounds__(kVScanThreads) v_scan_kernel(const float2* __restrict__ V, int64_t n,
                                                               float* __restrict__ amax_part,
                                                               double* __restrict__ Tpart, int32_t* status) {
  constexpr int NW = kVScanThreads / 32, kRows = R <= 4 ? 4 : 2;  // rows in flight per thread
  __shared__ double red[NW][2 * kMaxRank];
  __shared__ float wmax[NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double acc[2 * kMaxRank];
#pragma unroll
  for (int j = 0; j < 2 * kMaxRank; ++j) acc[j] = 0.0;
  float mx = 0.f;
  bool bad = false;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kVScanThreads;
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * kVScanThreads + threadIdx.x; i0 < n; i0 += kRows * stride) {
    float2 v[kRows][R];
#pragma unroll
    for (int q = 0; q < kRows; ++q)
#pragma unroll
      for (int j = 0; j < R; ++j)
        v[q][j] = i0 + q * stride < n ? V[(i0 + q * stride) * R + j] : make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kRows; ++q)
#pragma unroll
      for (int j = 0; j < R; ++j) {
        bad |= !isfinite(v[q][j].x) || !isfinite(v[q][j].y);
        mx = fmaxf(mx, fmaxf(fabsf(v[q][j].x), fabsf(v[q][j].y)));
        if (SUMS && i0 + q * stride < n) {
          acc[2 * j] += exact_double(v[q][j].x);
          acc[2 * j + 1] -= exact_double(v[q][j].y);
        }
      }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) dev_fail(status, LRQ_EINVAL);
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, m));
  if (lane == 0) wmax[warp] = mx;
  if (SUMS) {
    const double v = warp_sums16(acc);
    if ((lane & 1) == 0) red[warp][lane >> 1] = v;
  }
  __syncthreads();
  if (SUMS && threadIdx.x < 2 * R) {
    double v = red[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < NW; ++w) v += red[w][threadIdx.x];
    Tpart[static_cast<int64_t>(blockIdx.x) * 2 * kMaxRank + threadIdx.x] = v;
  }
  if (threadIdx.x == 0) {
    for (int w = 1; w < NW; ++w) mx = fmaxf(mx, wmax[w]);
    amax_part[blockIdx.x] = mx;
  }
}

// At most one block per SM; few rows a thread while that spreads them over more
// SMs (n = 3000, r = 4: 4.4 us, 15.1 with 2048 rows a block).
int v_scan_blocks(int64_t n) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kVScanMaxBlocks, ceil_div(n, kVScanThreads))));
}

int launch_v_scan(const float2* V, int64_t n, int r, bool sums, float* amax_part, double* Tpart, int32_t* status,
                  cudaStream_t st) {
  const int blocks = v_scan_blocks(n);
  switch (r) {
#define LRQ_VSCAN_CASE(RR)                                                                            \
  case RR:                                                                                            \
    if (sums)                                                                                         \
      v_scan_kernel<RR, true><<<blocks, kVScanThreads, 0, st>>>(V, n, amax_part, Tpart, status);      \
    else                                                                                              \
      v_scan_kernel<RR, false><<<blocks, kVScanThreads, 0, st>>>(V, n, amax_part, Tpart, status);     \
    break;
    LRQ_VSCAN_CASE(1)
    LRQ_VSCAN_CASE(2)
    LRQ_VSCAN_CASE(3)
    LRQ_VSCAN_CASE(4)
    LRQ_VSCAN_CASE(5)
    LRQ_VSCAN_CASE(6)
    LRQ_VSCAN_CASE(7)
    LRQ_VSCAN_CASE(8)
#undef LRQ_VSCAN_CASE
    default:
      return fail(LRQ_EUNSUPPORTED, "v_scan: r out of range");
  }
  count_launch();
  return cuda_check(cudaGetLastError(), "v_scan_kernel");
}

// ---------------------------------------------------------------------------
// FP32 CUDA-core scoring.
// Block: 256 candidates x one coordinate chunk (blockIdx.y).  Coordinates are
// staged through shared memory 256 rows at a time and read back as broadcasts.
// Per coordinate: w = V_i c (packed FP32 FMAs), decision from the boundary-line
// signs, V^H z += conj(V_i) omega^k (score_f32x2.cuh).  The FP32 running sum
// covers one 256-row batch and is then added into FP64 (blocked partials, so
// the FP32 error is that of a 256-term sum).
// Bound: the FMA pipe (38 cycles an evaluation at r = 4, K = 8) and the
// shared-memory reads.  The scalar form with one candidate a thread issued
// about 81 instructions an evaluation.  n = 4096, S = 2^14, r = 4, K = 8: 112
// us, 145 before (same bits).  Two candidates a thread while that leaves 16
// warps an SM; four halve the reads again but leave 12 warps here: 133 us.
// Output: partial[chunk][s][2r] doubles = (Re, Im) of sum_{i in chunk} conj(V_i) z_i.
// ---------------------------------------------------------------------------
struct Fp32Tables {
  float zr[kMaxK], zi[kMaxK];
};

constexpr int kFp32Block = 256;    // candidates
constexpr int kFp32Batch = 256;

template <int K, int R, int kFp32Cpt>  // kFp32Cpt: candidates per thread
__global__ void __launch_bounds__(kFp32Block / kFp32Cpt) score_fp32_kernel(const float2* __restrict__ V, int64_t n,
                                                                  const float2* __restrict__ C, int64_t S,
                                                                  int64_t S_pad, int64_t rows_per_chunk, int Kdyn,
                                                                  const __grid_constant__ Fp32Tables tab,
                                                                  double* __restrict__ partial) {
  constexpr int kFp32Threads = kFp32Block / kFp32Cpt;
  constexpr bool kScalar = K == 0;  // score_row_scalar
  __shared__ __align__(16) float4 vs[kScalar ? kFp32Batch * R / 2 : kFp32Batch * R];
  __shared__ float2 zt[ZTable<K>::kEntries];
  fill_ztable<K>(zt, tab.zr, tab.zi, Kdyn);

  const float none[kAnyLines] = {};  // the boundaries of kAnyK8, not used here
  const int64_t s0 = static_cast<int64_t>(blockIdx.x) * kFp32Block + threadIdx.x;
  Dir2<R> d[kFp32Cpt];
  float2 c[R];  // kScalar's
  double acc64[kFp32Cpt][2 * R];
#pragma unroll
  for (int q = 0; q < kFp32Cpt; ++q) {
    const int64_t s = s0 + q * kFp32Threads;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      c[j] = s < S ? C[s * R + j] : make_float2(0.f, 0.f);
      d[q].set(j, c[j]);
    }
#pragma unroll
    for (int j = 0; j < 2 * R; ++j) acc64[q][j] = 0.0;
  }

  const int64_t i_begin = static_cast<int64_t>(blockIdx.y) * rows_per_chunk;
  const int64_t i_end = min(n, i_begin + rows_per_chunk);
  for (int64_t b0 = i_begin; b0 < i_end; b0 += kFp32Batch) {
    const int rows = static_cast<int>(min(static_cast<int64_t>(kFp32Batch), i_end - b0));
    __syncthreads();
#pragma unroll 4
    for (int t = threadIdx.x; t < rows * R; t += kFp32Threads) {
      const float2 v = V[b0 * R + t];
      if constexpr (kScalar)
        reinterpret_cast<float2*>(vs)[t] = v;
      else
        vs[t] = make_float4(v.x, v.x, v.y, v.y);
    }
    __syncthreads();
    if constexpr (kScalar) {
      static_assert(kFp32Cpt == 1, "one candidate a thread");
      float2 acc[R];
#pragma unroll
      for (int j = 0; j < R; ++j) acc[j] = make_float2(0.f, 0.f);
      // four rows unrolled keep more angles in flight (n = 2000, r = 3: 73 us, 81 rolled);
      // at r = 4 the registers for it cost a block an SM (269 us, 261 with two)
#pragma unroll(R == 4 ? 2 : 4)
      for (int i = 0; i < rows; ++i) {
        float2 v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = reinterpret_cast<const float2*>(vs)[i * R + j];
        score_row_scalar<R, true>(v, c, zt, Kdyn, acc);
      }
#pragma unroll
      for (int j = 0; j < R; ++j) {
        acc64[0][2 * j] += static_cast<double>(acc[j].x);
        acc64[0][2 * j + 1] += static_cast<double>(acc[j].y);
      }
    } else {
      f32x2 acc[kFp32Cpt][R];
#pragma unroll
      for (int q = 0; q < kFp32Cpt; ++q)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[q][j] = 0;
      for (int i = 0; i < rows; ++i) {
        ulonglong2 v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = reinterpret_cast<const ulonglong2*>(vs)[i * R + j];
#pragma unroll
        for (int q = 0; q < kFp32Cpt; ++q) score_row<K, R, true>(v, d[q], zt, Kdyn, none, none, acc[q]);
      }
#pragma unroll
      for (int q = 0; q < kFp32Cpt; ++q)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          float re, im;
          unpack2(acc[q][j], re, im);
          acc64[q][2 * j] += static_cast<double>(re);
          acc64[q][2 * j + 1] += static_cast<double>(im);
        }
    }
  }
#pragma unroll
  for (int q = 0; q < kFp32Cpt; ++q) {
    const int64_t s = s0 + q * kFp32Threads;
    if (s < S) {
      double* out = partial + (static_cast<int64_t>(blockIdx.y) * S_pad + s) * (2 * R);
#pragma unroll
      for (int j = 0; j < 2 * R; ++j) out[j] = acc64[q][j];
    }
  }
}

// Two candidates a thread up to r = 5 and K = 8, once the blocks go round the chip
// several times: below that a thread's chain of evaluations is the time.  Kernel
// time with one / two: 4 blocks (K = 2, r = 1) 11 / 26 us, 160 (K = 8, r = 3) 34 / 42,
// 320 (K = 2, r = 4) 42 / 46, 1024 (K = 8, r = 4) 118 / 116, 1185 (K = 2, r = 3) 601 /
// 575.
template <int K, int R>
static void launch_fp32_one(const ScorePlan& p, dim3 grid, const Fp32Tables& tab, const float2* V, const float2* C,
                            double* partial, cudaStream_t st) {
  const int64_t S_pad = p.c_tiles * 128;
  const int64_t blocks = static_cast<int64_t>(grid.x) * grid.y;
  if constexpr (R <= 5 && K > 0) {
    if (blocks >= 4 * static_cast<int64_t>(num_sms_current())) {
      score_fp32_kernel<K, R, 2><<<grid, kFp32Block / 2, 0, st>>>(V, p.n, C, p.S, S_pad, p.fp32_rows_per_chunk, p.K, tab,
                                                                  partial);
      return;
    }
  }
  score_fp32_kernel<K, R, 1><<<grid, kFp32Block, 0, st>>>(V, p.n, C, p.S, S_pad, p.fp32_rows_per_chunk, p.K, tab,
                                                          partial);
}

template <int K>
static int launch_fp32_r(const ScorePlan& p, const Fp32Tables& tab, const float2* V, const float2* C,
                         double* partial, cudaStream_t st) {
  dim3 grid(static_cast<unsigned>(ceil_div(p.S, kFp32Block)), static_cast<unsigned>(p.nsplit));
  switch (p.r) {
#define LRQ_FP32_CASE(RR)                                       \
  case RR:                                                      \
    launch_fp32_one<K, RR>(p, grid, tab, V, C, partial, st);    \
    break;
    LRQ_FP32_CASE(1)
    LRQ_FP32_CASE(2)
    LRQ_FP32_CASE(3)
    LRQ_FP32_CASE(4)
    LRQ_FP32_CASE(5)
    LRQ_FP32_CASE(6)
    LRQ_FP32_CASE(7)
    LRQ_FP32_CASE(8)
#undef LRQ_FP32_CASE
    default:
      return fail(LRQ_EUNSUPPORTED, "score_fp32: r out of range");
  }
  count_launch();
  return cuda_check(cudaGetLastError(), "score_fp32_kernel");
}

int launch_score_fp32(const ScorePlan& p, const Alphabet& a, const float2* V, const float2* C,
                      double* partial, cudaStream_t st) {
  Fp32Tables tab;
  for (int k = 0; k < kMaxK; ++k) {
    tab.zr[k] = k < a.K ? a.zr[k] : 0.f;
    tab.zi[k] = k < a.K ? a.zi[k] : 0.f;
  }
  switch (p.K) {
    case 2: return launch_fp32_r<2>(p, tab, V, C, partial, st);
    case 3: return launch_fp32_r<3>(p, tab, V, C, partial, st);
    case 4: return launch_fp32_r<4>(p, tab, V, C, partial, st);
    case 5: return launch_fp32_r<5>(p, tab, V, C, partial, st);
    case 6: return launch_fp32_r<6>(p, tab, V, C, partial, st);
    case 7: return launch_fp32_r<7>(p, tab, V, C, partial, st);
    case 8: return launch_fp32_r<8>(p, tab, V, C, partial, st);
    default: return launch_fp32_r<0>(p, tab, V, C, partial, st);
  }
}

// ---------------------------------------------------------------------------
// Finalisation: add the chunk partials in FP64 (in chunk order), add the base
// T for the odd-K indicator form, f = ||.||^2.  Writes the FP32 score and the
// selection key (score bits above the complemented index: larger key = larger
// f, ties to the smaller index).
// ---------------------------------------------------------------------------
// A thread per (candidate, component) adds the chunk partials (coalesced
// reads, 2r times as many threads as candidates), then one per candidate forms
// f.  A thread per candidate took 14.5 us at S = 2^14, 16 chunks, r = 4, 7.6
// now; same additions in the same order.
constexpr int kFinThreads = 256;

__global__ void __launch_bounds__(kFinThreads) finalize_kernel(const double* __restrict__ partial, int nsplit,
                                                               int64_t S, int64_t S_pad, int r2,
                                                               const double* __restrict__ T,
                                                               float* __restrict__ scores, uint64_t* __restrict__ keys) {
  __shared__ double vj[kFinThreads];
  const int per = kFinThreads / r2;  // candidates per block
  const int c = threadIdx.x / r2, j = threadIdx.x - c * r2;
  const int64_t s0 = static_cast<int64_t>(blockIdx.x) * per;
  double v = 0.0;
  if (c < per && s0 + c < S) {
    v = T ? T[j] : 0.0;
    const double* src = partial + (s0 + c) * r2 + j;
#pragma unroll 4
    for (int k = 0; k < nsplit; ++k) v += src[static_cast<int64_t>(k) * S_pad * r2];
  }
  vj[threadIdx.x] = v;
  __syncthreads();
  const int64_t s = s0 + threadIdx.x;
  if (static_cast<int>(threadIdx.x) >= per || s >= S) return;
  double f = 0.0;
  for (int q = 0; q < r2; ++q) {
    const double x = vj[threadIdx.x * r2 + q];
    f += x * x;
  }
  const float ff = static_cast<float>(f);
  if (scores) scores[s] = ff;
  if (keys)
    keys[s] = (static_cast<uint64_t>(__float_as_uint(ff)) << 32) |
              static_cast<uint64_t>(0xFFFFFFFFu - static_cast<uint32_t>(s));
}

int launch_finalize(const ScorePlan& p, const double* partial, const double* T, float* scores, uint64_t* keys,
                    cudaStream_t st) {
  const int per = kFinThreads / (2 * p.r);
  finalize_kernel<<<static_cast<unsigned>(ceil_div(p.S, per)), kFinThreads, 0, st>>>(
      partial, p.npart, p.S, p.c_tiles * 128, 2 * p.r, T, scores, keys);
  count_launch();
  return cuda_check(cudaGetLastError(), "finalize_kernel");
}

}  // namespace lrq
