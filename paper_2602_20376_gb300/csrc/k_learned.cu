// k_learned.cu -- the learned proposal: spectral features, a 3-layer MLP
// (forward, backward, Adam), and a mixture of von Mises-Fisher densities on
// S^7 (negative log-likelihood with its gradient, and sampling).  The paper
// has no learned component; the sampling it replaces is uniform on the
// sphere (Sec. 4.2), and the K-fold equivalence of directions (Sec. 2.3)
// lets targets live in one canonical window.
//
// Layouts: V is B x n x r complex64 (instance-major); parameters are one
// flat FP32 array W1 (F x 256), b1, W2 (256 x 256), b2, W3 (256 x 160), b3,
// each W row-major (in x out) so that a layer is y = x W + b.  In BF16 mode
// every GEMM operand is rounded to bfloat16 (round to nearest even) as it is
// staged in shared memory and the products accumulate in FP32, on the tensor
// cores (k_mlp_tc.cu); FP32 mode runs the CUDA-core GEMM below.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "gauss_df32.cuh"
#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

namespace cg = cooperative_groups;

constexpr int kWidth = 256;
constexpr int kComp = 16;
constexpr int kHead = 10;
constexpr int kOut = kComp * kHead;  // 160
constexpr int kDim = 8;              // S^7 in R^8 = C^4

// ---------------------------------------------------------------------------
// features (FP64): gauge, then eigenvalue shares and moments
// ---------------------------------------------------------------------------
__device__ __forceinline__ df32 df_from(double x) {
  const float h = static_cast<float>(x);
  return df32{h, static_cast<float>(x - static_cast<double>(h))};
}

// A cluster of blocks per instance, each with every NB-th group of 256 rows.
// Two passes over V: the entries of largest modulus and the sums of the row
// norms and column moduli; then the gauge-fixed copy and the central moments
// of all r + 1 populations at once (q = 0: a_i = ||V_i||^2 n / total, q = 1 + j:
// b_ij = |V_ij|^2 n / lambda_j).  Bound: FP64 (about 60 warp instructions of 16
// cycles per 32 rows at r = 4); the gauge product is double-float, in FP64 where
// its rounding to FP32 could depend on that.  One block
// per instance with eleven passes took 247 us at B = 16, n = 4096; 77 now.
constexpr int kFeatThreads = 256;
constexpr int kFeatSums = 3 * (kMaxRank + 1);

struct FeatShared {
  double part[kFeatThreads / 32][kFeatSums];
  double sum[kFeatSums];            // the block's sums, then the cluster's
  long long best[kMaxRank];         // bits of the largest |V_ij|^2 (non-negative doubles order like their bits)
  long long row[kMaxRank];
  long long wbest[kFeatThreads / 32][kMaxRank], wrow[kFeatThreads / 32][kMaxRank];
  df32 ph_re[kMaxRank], ph_im[kMaxRank];
  double ph_re64[kMaxRank], ph_im64[kMaxRank];
};

// the cluster's sums of `count` values per thread, in a fixed order
__device__ __forceinline__ void feat_sums(cg::cluster_group& cluster, FeatShared& sh, const double* v, int count) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int q = 0; q < count; ++q) {
    double s = v[q];
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    if (lane == 0) sh.part[warp][q] = s;
  }
  __syncthreads();
  double mine = 0.0;
  if (threadIdx.x < count)
    for (int w = 0; w < kFeatThreads / 32; ++w) mine += sh.part[w][threadIdx.x];
  if (threadIdx.x < count) sh.sum[threadIdx.x] = mine;
  cluster.sync();
  double total = 0.0;
  if (threadIdx.x < count)
    for (int b = 0; b < static_cast<int>(cluster.num_blocks()); ++b)
      total += cluster.map_shared_rank(&sh.sum[0], b)[threadIdx.x];
  cluster.sync();  // every block has read the others' sums
  if (threadIdx.x < count) sh.sum[threadIdx.x] = total;
  __syncthreads();
}

__device__ __forceinline__ double feat_mod2(float2 v) {
  return fma(static_cast<double>(v.x), static_cast<double>(v.x), static_cast<double>(v.y) * static_cast<double>(v.y));
}

__global__ void __launch_bounds__(kFeatThreads) features_kernel(const float2* __restrict__ V, int64_t n, int r,
                                                                const double* __restrict__ lambda,
                                                                float2* __restrict__ Vg, float* __restrict__ feat,
                                                                int32_t* status) {
  __shared__ FeatShared sh;
  cg::cluster_group cluster = cg::this_cluster();
  const int nb = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  const int b = blockIdx.x / nb;
  const float2* Vb = V + static_cast<int64_t>(b) * n * r;
  const double* lam = lambda + static_cast<int64_t>(b) * r;
  const int F = 5 * r + 4;
  float* fo = feat + static_cast<int64_t>(b) * F;
  double total = 0.0;
  for (int j = 0; j < r; ++j) total += lam[j];
  if (!(total > 0.0)) {  // the same for every block of the cluster
    if (threadIdx.x == 0 && rank == 0) dev_fail(status, LRQ_EINVAL);
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i0 = static_cast<int64_t>(rank) * kFeatThreads + threadIdx.x, stride = static_cast<int64_t>(nb) * kFeatThreads;
  double scale[kMaxRank + 1], acc[kFeatSums];
  scale[0] = static_cast<double>(n) / total;
#pragma unroll
  for (int j = 0; j < kMaxRank; ++j) scale[1 + j] = j < r ? static_cast<double>(n) / lam[j] : 0.0;
#pragma unroll
  for (int q = 0; q < kFeatSums; ++q) acc[q] = 0.0;
  // pass 1: per column the entry of largest modulus (lowest row on ties), sums
  long long best[kMaxRank], brow[kMaxRank];
#pragma unroll
  for (int j = 0; j < kMaxRank; ++j) {
    best[j] = -1;
    brow[j] = n;
  }
  for (int64_t i = i0; i < n; i += stride) {
    double a = 0.0;
#pragma unroll
    for (int j = 0; j < kMaxRank; ++j) {
      if (j < r) {
        const double m2 = feat_mod2(Vb[i * r + j]);
        const long long bits = __double_as_longlong(m2);
        if (m2 == m2 && bits > best[j]) {
          best[j] = bits;
          brow[j] = i;
        }
        a += m2;
        acc[1 + j] = fma(m2, scale[1 + j], acc[1 + j]);
      }
    }
    acc[0] = fma(a, scale[0], acc[0]);
  }
  auto better = [](long long& v, long long& row, long long o, long long orow) {
    if (o > v || (o == v && orow < row)) {
      v = o;
      row = orow;
    }
  };
#pragma unroll
  for (int j = 0; j < kMaxRank; ++j) {
    if (j < r) {
#pragma unroll
      for (int m = 16; m > 0; m >>= 1)
        better(best[j], brow[j], __shfl_xor_sync(0xffffffffu, best[j], m), __shfl_xor_sync(0xffffffffu, brow[j], m));
      if (lane == 0) {
        sh.wbest[warp][j] = best[j];
        sh.wrow[warp][j] = brow[j];
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < r) {
    long long v = sh.wbest[0][threadIdx.x], row = sh.wrow[0][threadIdx.x];
    for (int w = 1; w < kFeatThreads / 32; ++w) better(v, row, sh.wbest[w][threadIdx.x], sh.wrow[w][threadIdx.x]);
    sh.best[threadIdx.x] = v;
    sh.row[threadIdx.x] = row;
  }
  cluster.sync();
  if (threadIdx.x < r) {
    const int j = threadIdx.x;
    long long v = -1, row = n;
    for (int q = 0; q < nb; ++q)
      better(v, row, cluster.map_shared_rank(&sh.best[0], q)[j], cluster.map_shared_rank(&sh.row[0], q)[j]);
    const float2 a = Vb[min(row, static_cast<long long>(n - 1)) * r + j];
    const double am = sqrt(static_cast<double>(a.x) * a.x + static_cast<double>(a.y) * a.y);
    // multiply the column by |a| / a = conj(a) / |a|
    sh.ph_re64[j] = am > 0.0 ? a.x / am : 1.0;
    sh.ph_im64[j] = am > 0.0 ? -a.y / am : 0.0;
    sh.ph_re[j] = df_from(sh.ph_re64[j]);
    sh.ph_im[j] = df_from(sh.ph_im64[j]);
  }
  feat_sums(cluster, sh, acc, r + 1);  // its barriers also publish the phases
  double mean[kMaxRank + 1];
#pragma unroll
  for (int q = 0; q <= kMaxRank; ++q) mean[q] = q <= r ? sh.sum[q] / static_cast<double>(n) : 0.0;
#pragma unroll
  for (int q = 0; q < kFeatSums; ++q) acc[q] = 0.0;
  // pass 2: gauge-fixed copy, central moments
  float2* Vo = Vg + static_cast<int64_t>(b) * n * r;
  auto moments = [&](int q, double x) {
    const double d = fma(x, scale[q], -mean[q]), d2 = d * d;
    acc[3 * q] += d2;
    acc[3 * q + 1] = fma(d2, d, acc[3 * q + 1]);
    acc[3 * q + 2] = fma(d2, d2, acc[3 * q + 2]);
  };
  for (int64_t i = i0; i < n; i += stride) {
    double a = 0.0;
#pragma unroll
    for (int j = 0; j < kMaxRank; ++j) {
      if (j < r) {
        const float2 v = Vb[i * r + j];
        const df32 pr = sh.ph_re[j], pi = sh.ph_im[j];
        const df32 x = df_times(df32{v.x, 0.f}, pr), y = df_times(df32{v.y, 0.f}, pi);
        const df32 z = df_times(df32{v.x, 0.f}, pi), w = df_times(df32{v.y, 0.f}, pr);
        const df32 re = df_sum(x, df32{-y.h, -y.l}), im = df_sum(z, w);
        float2 o = make_float2(re.h, im.h);
        // each product and sum is off by less than 2^-45 of the terms: where that
        // could turn the rounding (one entry in 10^5), in FP64
        const float err = 0x1p-43f * (fabsf(v.x) + fabsf(v.y));
        if (df_near_midpoint(re, err) || df_near_midpoint(im, err)) {
          o.x = static_cast<float>(v.x * sh.ph_re64[j] - v.y * sh.ph_im64[j]);
          o.y = static_cast<float>(v.x * sh.ph_im64[j] + v.y * sh.ph_re64[j]);
        }
        Vo[i * r + j] = o;
        const double m2 = feat_mod2(v);
        a += m2;
        moments(1 + j, m2);
      }
    }
    moments(0, a);
  }
  feat_sums(cluster, sh, acc, 3 * (r + 1));
  if (rank == 0) {
    if (threadIdx.x < r) fo[threadIdx.x] = static_cast<float>(lam[threadIdx.x] / total);
    if (threadIdx.x <= r) {
      const int q = threadIdx.x;
      const double dn = static_cast<double>(n);
      const double var = sh.sum[3 * q] / dn, m3 = sh.sum[3 * q + 1] / dn, m4 = sh.sum[3 * q + 2] / dn;
      double mq = 0.0;
#pragma unroll
      for (int k = 0; k <= kMaxRank; ++k)
        if (k == q) mq = mean[k];
      float* o = fo + r + 4 * q;
      o[0] = static_cast<float>(mq);
      o[1] = static_cast<float>(var);
      o[2] = var > 0.0 ? static_cast<float>(m3 / (var * sqrt(var))) : 0.f;
      o[3] = var > 0.0 ? static_cast<float>(m4 / (var * var) - 3.0) : 0.f;
    }
  }
}

// ---------------------------------------------------------------------------
// GEMM for the MLP: C = act(op(A) op(B) + bias) [* mask > 0]
//   op(A): M x K (A stored M x K, or K x M when ta), op(B): K x N (B stored
//   K x N, or N x K when tb).  32 x 32 tiles, 256 threads, 2 x 2 per thread.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__global__ void __launch_bounds__(256) mlp_gemm_kernel(int M, int N, int K, const float* __restrict__ A, int lda,
                                                       int ta, const float* __restrict__ Bm, int ldb, int tb,
                                                       const float* __restrict__ bias, int relu,
                                                       const float* __restrict__ mask, float* __restrict__ C,
                                                       int ldc, int bf16) {
  __shared__ float As[32][33], Bs[32][33];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row0 = blockIdx.y * 32, col0 = blockIdx.x * 32;
  float acc[2][2] = {{0.f, 0.f}, {0.f, 0.f}};
  for (int k0 = 0; k0 < K; k0 += 32) {
    for (int t = threadIdx.x; t < 32 * 32; t += 256) {
      const int i = t >> 5, k = t & 31;
      const int gr = row0 + i, gk = k0 + k;
      float a = 0.f;
      if (gr < M && gk < K) a = ta ? A[static_cast<int64_t>(gk) * lda + gr] : A[static_cast<int64_t>(gr) * lda + gk];
      As[i][k] = bf16 ? bf16_round(a) : a;
      const int gc = col0 + i;  // reuse i as the column for B
      float bv = 0.f;
      if (gc < N && gk < K) bv = tb ? Bm[static_cast<int64_t>(gc) * ldb + gk] : Bm[static_cast<int64_t>(gk) * ldb + gc];
      Bs[k][i] = bf16 ? bf16_round(bv) : bv;
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float a0 = As[ty * 2][k], a1 = As[ty * 2 + 1][k];
      const float b0 = Bs[k][tx * 2], b1 = Bs[k][tx * 2 + 1];
      acc[0][0] = fmaf(a0, b0, acc[0][0]);
      acc[0][1] = fmaf(a0, b1, acc[0][1]);
      acc[1][0] = fmaf(a1, b0, acc[1][0]);
      acc[1][1] = fmaf(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int gr = row0 + ty * 2 + u, gc = col0 + tx * 2 + v;
      if (gr >= M || gc >= N) continue;
      float x = acc[u][v] + (bias ? bias[gc] : 0.f);
      if (relu) x = fmaxf(x, 0.f);
      if (mask && !(mask[static_cast<int64_t>(gr) * ldc + gc] > 0.f)) x = 0.f;
      C[static_cast<int64_t>(gr) * ldc + gc] = x;
    }
}

// out[j] = sum_b G[b, j] (bias gradients), a thread per column, rows in order
__global__ void colsum_f32_kernel(const float* __restrict__ G, int B, int N, float* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  float s = 0.f;
  for (int b = 0; b < B; ++b) s += G[static_cast<int64_t>(b) * N + j];
  out[j] = s;
}

// ---------------------------------------------------------------------------
// vMF normaliser on S^7 (FP64): log I_nu by its power series for kappa <= 30
// and by the large-argument expansion above
// ---------------------------------------------------------------------------
// 1 / ((k + 1)(k + 1 + nu)), the ratio of consecutive series terms without
// (kappa / 2)^2: at kappa = 30 the terms fall below 1e-18 of the sum before
// k = 64, so 96 entries always suffice
constexpr int kBesselTerms = 96;
struct BesselTable {
  double v[2][kBesselTerms];  // nu = 3, 4
};
constexpr BesselTable make_bessel_table() {
  BesselTable t{};
  for (int h = 0; h < 2; ++h)
    for (int k = 0; k < kBesselTerms; ++k)
      t.v[h][k] = 1.0 / (static_cast<double>(k + 1) * static_cast<double>(k + 1 + 3 + h));
  return t;
}
__constant__ BesselTable c_bessel = make_bessel_table();

// log I_nu(kappa), nu = 3 + h
__device__ __forceinline__ double log_bessel_i_dev(int h, double kappa) {
  if (kappa <= 30.0) {
    const double half = 0.5 * kappa, h2 = half * half;
    double t = h == 0 ? h2 * half * (1.0 / 6.0) : h2 * h2 * (1.0 / 24.0);
    double s = t;
    for (int k = 0; k < kBesselTerms; ++k) {
      t *= h2 * c_bessel.v[h][k];
      s += t;
      if (t < 1e-18 * s) break;
    }
    return log(s);
  }
  const int nu = 3 + h;
  const double mu = 4.0 * nu * nu;
  const double ik = 1.0 / (8.0 * kappa);
  double s = 1.0, t = 1.0;
  for (int j = 1; j < 12; ++j) {
    const double o = 2.0 * j - 1.0;
    t *= -(mu - o * o) / j * ik;
    s += t;
  }
  return kappa - 0.5 * log(2.0 * kPi * kappa) + log(s);
}

struct CompParams {
  double mu[kComp][kDim];
  double unorm[kComp];
  double kappa[kComp];
  double sig[kComp];     // softplus'
  double logpi[kComp];
  double pi[kComp];
  double logc[kComp];
  double a8[kComp];
};

// Fills cp from one instance's outputs; every thread of the block calls it.
// One warp does the work: an SM's FP64 unit is two lanes wide, so a warp-wide
// FP64 instruction takes 16 cycles and what counts is how few of them there
// are.  Lanes m and m + 16 share component m (I_3 and I_4, half of mu each);
// the series multiply by tabulated reciprocals instead of dividing, and the
// weights are normalised across lanes instead of by one thread in turn
// (vmf_sample_kernel, which runs it once a block: 3092 -> 2298 us at B = 16,
// S = 65520).
__device__ void head_params(const float* __restrict__ O, CompParams& cp) {
  if (threadIdx.x < 32) {
    const int m = threadIdx.x & (kComp - 1), h = threadIdx.x >> 4;
    const float* o = O + m * kHead;
    double nrm = 0.0;
    for (int d = 0; d < kDim; ++d) nrm += static_cast<double>(o[d]) * o[d];
    nrm = sqrt(nrm);
    for (int d = h * (kDim / 2); d < (h + 1) * (kDim / 2); ++d)
      cp.mu[m][d] = nrm > 0.0 ? o[d] / nrm : (d == 0 ? 1.0 : 0.0);
    const double x = o[kDim];
    const double kap = x > 20.0 ? x : log1p(exp(x));
    const double li = log_bessel_i_dev(h, kap);
    const double li4 = __shfl_down_sync(0xffffffffu, li, 16);
    const double lg = o[kDim + 1];
    double mx = lg;
#pragma unroll
    for (int q = kComp / 2; q > 0; q >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, q));
    double s = exp(lg - mx);
#pragma unroll
    for (int q = kComp / 2; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if (h == 0) {
      cp.unorm[m] = nrm;
      cp.kappa[m] = kap;
      cp.sig[m] = 1.0 / (1.0 + exp(-x));
      cp.logc[m] = 3.0 * log(kap) - 4.0 * log(2.0 * kPi) - li;
      cp.a8[m] = exp(li4 - li);
      const double lp = lg - (mx + log(s));
      cp.logpi[m] = lp;
      cp.pi[m] = exp(lp);
    }
  }
  __syncthreads();
}

// Loss and gradient of the mean negative log-likelihood.  A cluster of NB
// blocks per instance, each taking every NB-th group of targets; a lane owns
// one component and half a warp one target, so that the 11 sums a component
// needs (of its responsibility gamma, gamma (mu.x - A_8), gamma mu.x and
// gamma x) stay in FP64 registers over all targets.  Bound: FP64 (about 60
// warp instructions of 16 cycles per 32 (target, component) pairs; 16 us of
// the whole chip at B = 64, T = 164).  The first version let every thread
// take a target and added 160 gradient terms per target into shared memory
// with FP64 atomics, all threads on the same address: 841 us at that size,
// now about 52.  The blocks' sums meet in shared memory (across the cluster) in a
// fixed order; the loss keeps its one atomic per block.
constexpr int kNllThreads = 128;
constexpr int kNllSums = 11;

// x's bits as an integer that orders like it: maxima run on the integer pipe
// (and the same map takes the integer back)
__device__ __forceinline__ long long order64(long long bits) {
  return bits >= 0 ? bits : bits ^ 0x7fffffffffffffffll;
}

__global__ void __launch_bounds__(kNllThreads) vmf_nll_kernel(const float* __restrict__ O, int B,
                                                              const float* __restrict__ X, int T,
                                                              double* __restrict__ loss, float* __restrict__ dO) {
  __shared__ CompParams cp;
  __shared__ double part[kNllThreads / 32][kNllSums][kComp];
  __shared__ double g[kNllSums][kComp];
  __shared__ double lred[kNllThreads / 16];
  cg::cluster_group cluster = cg::this_cluster();
  const int nb = static_cast<int>(cluster.num_blocks()), rank = static_cast<int>(cluster.block_rank());
  const int b = blockIdx.x / nb;
  const float* Ob = O + static_cast<int64_t>(b) * kOut;
  head_params(Ob, cp);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, m = lane & (kComp - 1), half = threadIdx.x >> 4;
  constexpr int kHalves = kNllThreads / 16;
  double mu[kDim], sum[kNllSums];
#pragma unroll
  for (int d = 0; d < kDim; ++d) mu[d] = cp.mu[m][d];
#pragma unroll
  for (int q = 0; q < kNllSums; ++q) sum[q] = 0.0;
  const double base = cp.logpi[m] + cp.logc[m], kap = cp.kappa[m], a8 = cp.a8[m];
  // -sum_t (shift_t + log se_t), the logarithm taken of products of se_t in
  // [1, 16]: 64 of them stay far inside the range
  double lsum = 0.0, prod = 1.0;
  int nprod = 0;
  const int groups = (T + kHalves - 1) / kHalves;
  const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0;  // rows are 32 bytes
  for (int gr = rank; gr < groups; gr += nb) {  // the same trips for every thread
    const int t = gr * kHalves + half;
    const bool act = t < T;
    const float4* x4 = reinterpret_cast<const float4*>(X + (static_cast<int64_t>(b) * T + (act ? t : T - 1)) * kDim);
    float xf[kDim];
    if (vec) {
      const float4 u = x4[0], w = x4[1];
      xf[0] = u.x, xf[1] = u.y, xf[2] = u.z, xf[3] = u.w, xf[4] = w.x, xf[5] = w.y, xf[6] = w.z, xf[7] = w.w;
    } else {
#pragma unroll
      for (int d = 0; d < kDim; ++d) xf[d] = reinterpret_cast<const float*>(x4)[d];
    }
    double xv[kDim], dot = 0.0;
#pragma unroll
    for (int d = 0; d < kDim; ++d) {
      xv[d] = xf[d];
      dot = fma(mu[d], xv[d], dot);
    }
    const double ell = fma(kap, dot, base);
    long long key = order64(__double_as_longlong(ell));
#pragma unroll
    for (int q = kComp / 2; q > 0; q >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, q));
    const double shift = __longlong_as_double(order64(key));
    const double e = exp(ell - shift);
    double se = e;
#pragma unroll
    for (int q = kComp / 2; q > 0; q >>= 1) se += __shfl_xor_sync(0xffffffffu, se, q);
    const double gam = act ? e / se : 0.0;
    if (act) {
      lsum -= shift;
      prod *= se;
    }
    if (++nprod == 64) {
      lsum -= log(prod);
      prod = 1.0;
      nprod = 0;
    }
    sum[0] += gam;
    sum[1] = fma(gam, dot - a8, sum[1]);
    sum[2] = fma(gam, dot, sum[2]);
#pragma unroll
    for (int d = 0; d < kDim; ++d) sum[3 + d] = fma(gam, xv[d], sum[3 + d]);
  }
  lsum -= log(prod);
  // the two halves of a warp, then the warps, then the blocks of the cluster
#pragma unroll
  for (int q = 0; q < kNllSums; ++q) {
    sum[q] += __shfl_xor_sync(0xffffffffu, sum[q], 16);
    if (lane < kComp) part[warp][q][m] = sum[q];
  }
  if (m == 0) lred[half] = lsum;
  __syncthreads();
  for (int k = threadIdx.x; k < kNllSums * kComp; k += kNllThreads) {
    double v = 0.0;
    for (int w = 0; w < kNllThreads / 32; ++w) v += part[w][k / kComp][k % kComp];
    g[k / kComp][k % kComp] = v;
  }
  const double inv = 1.0 / (static_cast<double>(B) * T);
  if (threadIdx.x == 0) {
    double ls = 0.0;
    for (int k = 0; k < kHalves; ++k) ls += lred[k];
    atomicAdd(loss, ls * inv);
  }
  cluster.sync();
  if (rank == 0) {
    for (int k = threadIdx.x; k < kNllSums * kComp; k += kNllThreads) {
      double v = g[k / kComp][k % kComp];
      for (int q = 1; q < nb; ++q) v += cluster.map_shared_rank(&g[0][0], q)[k];
      part[0][k / kComp][k % kComp] = v;
    }
    __syncthreads();
    // d/d logit = sum (pi - gamma), d/d kappa' = -softplus' sum gamma (mu.x - A_8),
    // d/d u = -(kappa / ||u||) (sum gamma x - mu sum gamma mu.x)
    for (int k = threadIdx.x; k < kOut; k += kNllThreads) {
      const int c = k / kHead, d = k % kHead;
      double v;
      if (d == kDim + 1)
        v = T * cp.pi[c] - part[0][0][c];
      else if (d == kDim)
        v = -cp.sig[c] * part[0][1][c];
      else
        v = -(cp.kappa[c] / cp.unorm[c]) * (part[0][3 + d][c] - cp.mu[c][d] * part[0][2][c]);
      dO[static_cast<int64_t>(b) * kOut + k] = static_cast<float>(v * inv);
    }
  }
  cluster.sync();  // the other blocks' sums stay until block 0 has read them
}

// ---------------------------------------------------------------------------
// sampling: component by its weight, Wood's rejection step for the cosine
// to mu, a uniform direction orthogonal to mu, then a random omega^k
//
// With G1, G2 the two Gamma(7/2) variates, b Wood's constant and
// Q = G2 + b G1 the candidate is w = (G2 - b G1) / Q, sqrt(1 - w^2) =
// 2 sqrt(b G1 G2) / Q (no cancellation at large kappa), and the acceptance test
//   kappa w + 7 log(1 - x0 w) - (kappa x0 + 7 log(1 - x0^2)) >= log u
// is 2 kappa b / (1 + b) (G2 - G1) / Q + 7 log((1 + b)(G1 + G2) / (2 Q)) >= log u.
// The test runs in FP32 with a margin; inside the margin (about one try in
// 10^4) it is repeated in FP64 as first written, so every draw is accepted or
// not as in FP64.  Logs, Gaussians and the vectors are double-float
// (gauss_df32.cuh): a component is within 2^-40 of FP64's before it is rounded to
// FP32 (of 960000 components 8 differ from numpy's FP64 rounding, 9 when all of it
// ran in FP64).  FP64 runs at 1/64 of the FP32 rate and took about 800
// instructions a sample (16 x 65520 draws: 2298 us, 361 with one sample a thread
// at a time).  A warp's tries run until its unluckiest lane is done, about four
// times where the mean is 1.5, so a thread takes kVmfPer samples through the
// tries one after the other and the warp then finishes all of them together:
// 262 us.
// ---------------------------------------------------------------------------
constexpr int kVmfThreads = 128;
constexpr int kVmfPer = 8;  // samples of a thread at a time

struct VmfRng {
  uint64_t seed;
  uint32_t s, b, ctr;
  // the two uniforms' 2 x + 1 over 2^54 (x: 53 bits)
  __device__ __forceinline__ void bits2(uint64_t* u, uint64_t* v) {
    const PhiloxOut o =
        philox4x32_10(s, b, ctr++, 0x564D46u, static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
    *u = ((((static_cast<uint64_t>(o.w[0]) << 32) | o.w[1]) >> 11) << 1) | 1ull;
    *v = ((((static_cast<uint64_t>(o.w[2]) << 32) | o.w[3]) >> 11) << 1) | 1ull;
  }
  __device__ double2 uniform2() {  // two 53-bit uniforms in (0, 1)
    PhiloxOut o = philox4x32_10(s, b, ctr++, 0x564D46u, static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
    return make_double2(uniform53(o.w[0], o.w[1]), uniform53(o.w[2], o.w[3]));
  }
  // Gamma(7/2) = Gamma(3) + Gamma(1/2): -log(u1 u2 u3) + n^2 / 2 with
  // n^2 / 2 = -log(u) cos^2
  __device__ __forceinline__ df32 gamma35() {
    uint64_t a, b2, c, d, e, f;
    bits2(&a, &b2);
    bits2(&c, &d);
    bits2(&e, &f);
    df32 sn, cs;
    df_sincos(f, GaussTab(), &sn, &cs);
    return df_sum(df_neg_log3(a, b2, c, GaussTab()), df_times(df_neg_log(e, GaussTab()), df_times(cs, cs)));
  }
  __device__ double gamma35_fp64() {
    const double2 a = uniform2(), c = uniform2(), u = uniform2();
    const double rad = sqrt(-2.0 * log(u.x));
    double sn, cs;
    sincospi(2.0 * u.y, &sn, &cs);
    return -log(a.x * a.y * c.x) + 0.5 * (rad * cs) * (rad * cs);
  }
};

// the acceptance test in FP64 for the try whose first counter is rng.ctr
__device__ __noinline__ bool vmf_accept_fp64(VmfRng rng, double kap, double bb, double x0, double cc) {
  const double g1 = rng.gamma35_fp64(), g2 = rng.gamma35_fp64();
  const double z = g1 / (g1 + g2);  // Beta(7/2, 7/2)
  const double w = (1.0 - (1.0 + bb) * z) / (1.0 - (1.0 - bb) * z);
  const double u = rng.uniform2().x;
  return kap * w + (kDim - 1.0) * log(1.0 - x0 * w) - cc >= log(u);
}

__global__ void __launch_bounds__(kVmfThreads) vmf_sample_kernel(const float* __restrict__ O, int B, int S, int K,
                                                                 int nper, uint64_t seed, float2* __restrict__ C,
                                                                 int32_t* status) {
  __shared__ CompParams cp;
  __shared__ double wb[kComp], wx0[kComp], wc[kComp];
  __shared__ long long cdf[kComp];  // bits of the cumulative weights (positive doubles order like their bits)
  __shared__ double total;
  __shared__ df32 smu[kComp][kDim], sb[kComp], root_c[kMaxK], root_s[kMaxK];
  __shared__ float sa[kComp], shalf[kComp];
  __shared__ float4 sw4[kVmfPer][kVmfThreads];    // w and sqrt(1 - w^2)
  __shared__ uint32_t smk[kVmfPer][kVmfThreads];  // component, power of omega
  __shared__ uint32_t sctr[kVmfPer][kVmfThreads]; // random numbers used
  const int b = blockIdx.y;
  head_params(O + static_cast<int64_t>(b) * kOut, cp);
  if (threadIdx.x < kComp) {
    const int m = threadIdx.x;
    const double kap = cp.kappa[m];
    const double p1 = kDim - 1.0;
    const double bb = p1 / (2.0 * kap + sqrt(4.0 * kap * kap + p1 * p1));  // = (-2k + sqrt(4k^2 + p1^2)) / p1
    const double x0 = (1.0 - bb) / (1.0 + bb);
    wb[m] = bb;
    wx0[m] = x0;
    wc[m] = kap * x0 + p1 * log(1.0 - x0 * x0);
    sb[m] = df_from(bb);
    sa[m] = static_cast<float>(2.0 * kap * bb / (1.0 + bb));
    shalf[m] = static_cast<float>(0.5 * (1.0 + bb));
  }
  for (int t = threadIdx.x; t < kComp * kDim; t += kVmfThreads) smu[t / kDim][t % kDim] = df_from(cp.mu[t / kDim][t % kDim]);
  if (threadIdx.x < K) {
    double sn, cs;
    sincospi(2.0 * threadIdx.x / static_cast<double>(K), &sn, &cs);
    root_c[threadIdx.x] = df_from(cs);
    root_s[threadIdx.x] = df_from(sn);
  }
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int m = 0; m < kComp; ++m) {
      s += cp.pi[m];
      cdf[m] = __double_as_longlong(s);
    }
    total = s;
  }
  __syncthreads();
  const int tid = threadIdx.x;
  for (int64_t b0 = static_cast<int64_t>(blockIdx.x) * kVmfThreads * nper; b0 < S;
       b0 += static_cast<int64_t>(gridDim.x) * kVmfThreads * nper) {
    const int base = static_cast<int>(b0) + tid;
    const int count = base < S ? min(nper, (S - 1 - base) / kVmfThreads + 1) : 0;
    for (int q = 0; q < count; ++q) {
      VmfRng rng{seed, static_cast<uint32_t>(base + q * kVmfThreads), static_cast<uint32_t>(b), 0u};
      uint64_t ux, uy;
      rng.bits2(&ux, &uy);
      // the component and the member of the K-fold equivalence class
      const long long target = __double_as_longlong((static_cast<double>(ux >> 1) + 0.5) * (1.0 / 9007199254740992.0) * total);
      int m = 0;
      while (m < kComp - 1 && cdf[m] < target) ++m;
      const int k = min(K - 1, static_cast<int>(__umul64hi(uy << 10, static_cast<uint64_t>(K))));
      smk[q][tid] = static_cast<uint32_t>(m) | static_cast<uint32_t>(k) << 8;
    }
    for (int q = 0, tries = 0, ctr = 1; q < count;) {
      VmfRng rng{seed, static_cast<uint32_t>(base + q * kVmfThreads), static_cast<uint32_t>(b), static_cast<uint32_t>(ctr)};
      const int m = smk[q][tid] & 0xffu;
      const VmfRng at = rng;
      const df32 bb = sb[m], g1 = rng.gamma35(), g2 = rng.gamma35();
      uint64_t u, unused;
      rng.bits2(&u, &unused);
      const df32 bg = df_times(bb, g1), sum = df_sum(g2, bg);
      const float rq = 1.0f / sum.h;
      const float t1 = sa[m] * ((g2.h - g1.h) + (g2.l - g1.l)) * rq;
      const float t2 = (kDim - 1.0f) * logf(shalf[m] * (g1.h + g2.h) * rq);
      const float lu = -df_neg_log(u, GaussTab()).h;
      const float d = t1 + t2 - lu;
      // FP32 rounding of terms of size |t1|, |t2|, |lu|: below 16 * 2^-24 each
      const float margin = 1e-5f * (1.0f + fabsf(t1) + fabsf(t2) + fabsf(lu));
      bool ok = d >= 0.0f;
      if (fabsf(d) <= margin) ok = vmf_accept_fp64(at, cp.kappa[m], wb[m], wx0[m], wc[m]);
      ctr = static_cast<int>(rng.ctr);
      if (!ok && ++tries < 1000) continue;
      if (!ok) dev_fail(status, LRQ_ETIMEOUT);
      const df32 r = df_recip(sum), w = df_times(df_sum(g2, df32{-bg.h, -bg.l}), r);
      const df32 root = df_times(df_sqrt(df_times(bg, g2)), r);
      sw4[q][tid] = make_float4(w.h, w.l, 2.0f * root.h, 2.0f * root.l);
      sctr[q][tid] = rng.ctr;
      ++q;
      tries = 0;
      ctr = 1;
    }
    __syncwarp();  // a thread reads its own entries; the warp goes on together
    for (int q = 0; q < count; ++q) {
      const int s = base + q * kVmfThreads, m = smk[q][tid] & 0xffu, k = smk[q][tid] >> 8;
      const float4 ws = sw4[q][tid];
      const df32 w{ws.x, ws.y}, sw{ws.z, ws.w};
      VmfRng rng{seed, static_cast<uint32_t>(s), static_cast<uint32_t>(b), sctr[q][tid]};
      // a Gaussian vector (up to its scale) made orthogonal to mu
      df32 v[kDim], dot{0.f, 0.f};
  #pragma unroll
      for (int d = 0; d < kDim; d += 2) {
        uint64_t e, f;
        rng.bits2(&e, &f);
        const df32 rad = df_sqrt(df_neg_log(e, GaussTab()));
        df32 sn, cs;
        df_sincos(f, GaussTab(), &sn, &cs);
        v[d] = df_times(rad, cs);
        v[d + 1] = df_times(rad, sn);
      }
  #pragma unroll
      for (int d = 0; d < kDim; ++d) dot = df_sum(dot, df_times(v[d], smu[m][d]));
      df32 nv{0.f, 0.f};
  #pragma unroll
      for (int d = 0; d < kDim; ++d) {
        const df32 t = df_times(dot, smu[m][d]);
        v[d] = df_sum(v[d], df32{-t.h, -t.l});
        nv = df_sum(nv, df_times(v[d], v[d]));
      }
      const df32 scale = nv.h > 0.f ? df_times(sw, df_recip(df_sqrt(nv))) : df32{0.f, 0.f};
      const df32 cs = root_c[k], sn = root_s[k];
      float2* out = C + (static_cast<int64_t>(b) * S + s) * (kDim / 2);
  #pragma unroll
      for (int j = 0; j < kDim / 2; ++j) {
        const df32 re = df_sum(df_times(w, smu[m][2 * j]), df_times(scale, v[2 * j]));
        const df32 im = df_sum(df_times(w, smu[m][2 * j + 1]), df_times(scale, v[2 * j + 1]));
        const df32 p = df_times(im, sn), q = df_times(im, cs);
        const df32 x = df_sum(df_times(re, cs), df32{-p.h, -p.l}), y = df_sum(df_times(re, sn), q);
        out[j] = make_float2(x.h, y.h);
      }
    }
  }
}

// The mixture's component means, ordered by weight (largest logit first,
// lower component index on ties): the most probable directions of the
// proposal, as directions of C^4.  A component with u = 0 gives e_1, the
// same convention as the sampler.  One warp per instance.
__global__ void vmf_modes_kernel(const float* __restrict__ O, int B, float2* __restrict__ C) {
  const int b = blockIdx.x;
  const int m = threadIdx.x;
  if (b >= B || m >= kComp) return;
  const float* Ob = O + static_cast<int64_t>(b) * kOut;
  const float lm = Ob[m * kHead + kDim + 1];
  int rank = 0;
  for (int k = 0; k < kComp; ++k) {
    const float lk = Ob[k * kHead + kDim + 1];
    rank += (lk > lm || (lk == lm && k < m)) ? 1 : 0;
  }
  double nrm = 0.0;
  for (int d = 0; d < kDim; ++d) nrm += static_cast<double>(Ob[m * kHead + d]) * Ob[m * kHead + d];
  nrm = sqrt(nrm);
  float2* out = C + (static_cast<int64_t>(b) * kComp + rank) * (kDim / 2);
  for (int j = 0; j < kDim / 2; ++j) {
    const double re = nrm > 0.0 ? Ob[m * kHead + 2 * j] / nrm : (j == 0 ? 1.0 : 0.0);
    const double im = nrm > 0.0 ? Ob[m * kHead + 2 * j + 1] / nrm : 0.0;
    out[j] = make_float2(static_cast<float>(re), static_cast<float>(im));
  }
}

// ---------------------------------------------------------------------------
// Adam (Kingma and Ba) with bias correction
// ---------------------------------------------------------------------------
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t count, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += stride) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
int64_t proposal_num_params(int F) {
  return static_cast<int64_t>(F) * kWidth + kWidth + kWidth * kWidth + kWidth + kWidth * kOut + kOut;
}

int launch_features(const float2* V, int B, int64_t n, int r, const double* lambda, float2* Vg, float* feat,
                    int32_t* status, cudaStream_t st) {
  // blocks per instance: about two per SM over all instances, a group of rows
  // each at least, at most the portable cluster size
  int nb = 1;
  while (nb < 8 && static_cast<int64_t>(B) * nb * 2 <= 2 * num_sms_current() && n > static_cast<int64_t>(nb) * kFeatThreads)
    nb *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(B) * nb);
  cfg.blockDim = dim3(kFeatThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nb;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const int e = cuda_check(cudaLaunchKernelEx(&cfg, features_kernel, V, n, r, lambda, Vg, feat, status),
                           "features_kernel");
  count_launch();
  return e;
}

// BF16 mode on the tensor cores (k_mlp_tc.cu); FP32 mode on the CUDA cores
static int gemm(cudaStream_t st, int M, int N, int K, const float* A, int lda, int ta, const float* Bm, int ldb,
                int tb, const float* bias, int relu, const float* mask, float* C, int ldc, int bf16) {
  if (bf16) return launch_mlp_gemm_tc(st, M, N, K, A, lda, ta, Bm, ldb, tb, bias, relu, mask, C, ldc);
  dim3 grid(static_cast<unsigned>(ceil_div(N, 32)), static_cast<unsigned>(ceil_div(M, 32)));
  mlp_gemm_kernel<<<grid, 256, 0, st>>>(M, N, K, A, lda, ta, Bm, ldb, tb, bias, relu, mask, C, ldc, 0);
  count_launch();
  return LRQ_OK;
}

int launch_mlp_forward(const float* params, int F, int B, const float* X, float* H1, float* H2, float* O, int bf16,
                       cudaStream_t st) {
  const float* W1 = params;
  const float* b1 = W1 + static_cast<int64_t>(F) * kWidth;
  const float* W2 = b1 + kWidth;
  const float* b2 = W2 + kWidth * kWidth;
  const float* W3 = b2 + kWidth;
  const float* b3 = W3 + kWidth * kOut;
  int e;
  if ((e = gemm(st, B, kWidth, F, X, F, 0, W1, kWidth, 0, b1, 1, nullptr, H1, kWidth, bf16))) return e;
  if ((e = gemm(st, B, kWidth, kWidth, H1, kWidth, 0, W2, kWidth, 0, b2, 1, nullptr, H2, kWidth, bf16))) return e;
  if ((e = gemm(st, B, kOut, kWidth, H2, kWidth, 0, W3, kOut, 0, b3, 0, nullptr, O, kOut, bf16))) return e;
  return cuda_check(cudaGetLastError(), "mlp forward");
}

int launch_mlp_backward(const float* params, int F, int B, const float* X, const float* H1, const float* H2,
                        const float* dO, float* grads, float* scratch, int bf16, cudaStream_t st) {
  const float* W2 = params + static_cast<int64_t>(F) * kWidth + kWidth;
  const float* W3 = W2 + kWidth * kWidth + kWidth;
  float* dW1 = grads;
  float* db1 = dW1 + static_cast<int64_t>(F) * kWidth;
  float* dW2 = db1 + kWidth;
  float* db2 = dW2 + kWidth * kWidth;
  float* dW3 = db2 + kWidth;
  float* db3 = dW3 + kWidth * kOut;
  float* dH2 = scratch;
  float* dH1 = scratch + static_cast<int64_t>(B) * kWidth;
  int e;
  // layer 3
  if ((e = gemm(st, kWidth, kOut, B, H2, kWidth, 1, dO, kOut, 0, nullptr, 0, nullptr, dW3, kOut, bf16))) return e;
  colsum_f32_kernel<<<1, 256, 0, st>>>(dO, B, kOut, db3);
  if ((e = gemm(st, B, kWidth, kOut, dO, kOut, 0, W3, kOut, 1, nullptr, 0, H2, dH2, kWidth, bf16))) return e;
  // layer 2
  if ((e = gemm(st, kWidth, kWidth, B, H1, kWidth, 1, dH2, kWidth, 0, nullptr, 0, nullptr, dW2, kWidth, bf16)))
    return e;
  colsum_f32_kernel<<<1, 256, 0, st>>>(dH2, B, kWidth, db2);
  if ((e = gemm(st, B, kWidth, kWidth, dH2, kWidth, 0, W2, kWidth, 1, nullptr, 0, H1, dH1, kWidth, bf16))) return e;
  // layer 1
  if ((e = gemm(st, F, kWidth, B, X, F, 1, dH1, kWidth, 0, nullptr, 0, nullptr, dW1, kWidth, bf16))) return e;
  colsum_f32_kernel<<<1, 256, 0, st>>>(dH1, B, kWidth, db1);
  count_launch(3);
  return cuda_check(cudaGetLastError(), "mlp backward");
}

int launch_vmf_nll(const float* O, int B, const float* X, int T, double* loss, float* dO, cudaStream_t st) {
  int e = cuda_check(cudaMemsetAsync(loss, 0, sizeof(double), st), "reset loss");
  if (e) return e;
  // blocks per instance: up to two per SM over all instances, at least two
  // groups of targets each, at most the portable cluster size
  int nb = 1;
  while (nb < 8 && static_cast<int64_t>(B) * nb * 2 <= 2 * 152 && T >= 4 * nb * (kNllThreads / 16)) nb *= 2;
  if (B > 0x7fffffff / nb) return fail(LRQ_EUNSUPPORTED, "vmf_nll: batch too large");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(B) * nb);
  cfg.blockDim = dim3(kNllThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nb;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cuda_check(cudaLaunchKernelEx(&cfg, vmf_nll_kernel, O, B, X, T, loss, dO), "vmf_nll_kernel");
  count_launch();
  return e;
}

int launch_vmf_sample(const float* O, int B, int S, int K, uint64_t seed, float2* C, int32_t* status,
                      cudaStream_t st) {
  // about eight blocks per SM over all instances (a block works out its
  // instance's parameters once, a few us of FP64), then several samples a thread
  const int64_t want = static_cast<int64_t>(8) * num_sms_current();
  const int nper = static_cast<int>(
      std::min<int64_t>(kVmfPer, std::max<int64_t>(1, ceil_div(static_cast<int64_t>(S) * B, want * kVmfThreads))));
  const int64_t per = std::max<int64_t>(1, ceil_div(want, B));
  dim3 grid(static_cast<unsigned>(std::min<int64_t>(ceil_div(S, kVmfThreads * nper), per)), static_cast<unsigned>(B));
  vmf_sample_kernel<<<grid, kVmfThreads, 0, st>>>(O, B, S, K, nper, seed, C, status);
  count_launch();
  return cuda_check(cudaGetLastError(), "vmf_sample_kernel");
}

int launch_vmf_modes(const float* O, int B, float2* C, cudaStream_t st) {
  vmf_modes_kernel<<<B, 32, 0, st>>>(O, B, C);
  count_launch();
  return cuda_check(cudaGetLastError(), "vmf_modes_kernel");
}

int launch_adam(float* p, const float* g, float* m, float* v, int64_t count, int t, float lr, float b1, float b2,
                float eps, cudaStream_t st) {
  const float c1 = 1.f - powf(b1, static_cast<float>(t)), c2 = 1.f - powf(b2, static_cast<float>(t));
  const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(count, 256), 152 * 8));
  adam_kernel<<<blocks, 256, 0, st>>>(p, g, m, v, count, lr, b1, b2, eps, c1, c2);
  count_launch();
  return cuda_check(cudaGetLastError(), "adam_kernel");
}

}  // namespace lrq
