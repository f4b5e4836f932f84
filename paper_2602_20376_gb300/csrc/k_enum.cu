// k_enum.cu -- exact rank-r solver by vertex enumeration of the hyperplane
// arrangement (Sec. 3, Algorithm 2; Theorem 3.2).
//
// Level d = r, r-1, ..., 1 uses the leading columns V[:, :d] (the recursion of
// Algorithm 2).  The augmented real matrix (Eq. 6) has rows
//   h_(i,m) = [Im(rho_m V_i), Re(rho_m V_i)],  rho_m = exp(-i pi (2m+1)/K),
// m < B_K, so that h . [Re c; Im c] = Im(rho_m V_i c) vanishes exactly when
// V_i c lies on decision boundary m.  For every index set I of 2d-1 rows with
// at most two rows from any coordinate group:
//   1. the null vector c~ of H_I (FP64 Gaussian elimination with full
//      pivoting; I is skipped unless H_I has rank 2d-1);
//   2. for both signs, c = +-(c~[:d] + i c~[d:]) and w = V_d c;
//   3. every coordinate gets the codes of the cells that touch the vertex: all
//      K codes where w_i = 0 (two rows of its group in I), both codes next to
//      the boundary where arg w_i is within 1e-9 of one, else the decision-rule
//      code (Eq. 9);
//   4. every combination is scored on the full V (||V^H z||^2), incrementally
//      from the all-decided base sum.
// Step 3 is a superset of the candidates of the paper's ambiguity resolution
// (Algorithm 4): every cell of the arrangement has a vertex in its closure.
// GB300's FP64 rate is 1/64 of its FP32 rate, so step 4 in FP64 is kept for
// the vertices that can win.  A block takes kEnumChunk consecutive index sets;
// for each, a thread finds the null vector in FP64 (the rank test decides
// which sets count) and evaluates both signs in FP32 with rigorous error
// bounds: f_up, an upper bound of every candidate of the vertex.  A vertex
// whose f_up is below the best FP64 value found so far anywhere holds no
// candidate that could win or tie; a vertex whose FP32 decisions are not
// certain is passed on whatever its value.  What is passed on is evaluated in
// FP64 as the steps above say, the block's largest f_up first, so the result
// (value, order of ties, error reports) is that of evaluating every vertex in
// FP64.  n = 64, r = 2, K = 3 (1.16 * 10^6 sets): 42.4 ms when every vertex
// was, 2.5 to 3.1 ms by instance now.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "enum_device.cuh"
#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

constexpr int kEnumMaxN = 512;
constexpr int kEnumThreads = 128;
constexpr int kEnumRanksPerThread = 16;                         // at most
constexpr int kEnumChunk = kEnumThreads * kEnumRanksPerThread;  // index sets per block step, at most
constexpr int kEnumBlocks = 4096;                               // at most, per level
constexpr double kEnumDefaultBudget = 1e12;

// The FP32 copy of V (a power of two brings its largest component into
// [1, 2)) and what the error bounds need.
struct EnumF32 {
  float zr[kMaxTcK], zi[kMaxTcK];      // omega^k
  float bcos[kMaxTcK], bsin[kMaxTcK];  // all K boundaries
};
struct EnumScan {
  double scale;  // V32 = V scale
  float esum;    // bound of the error of |V^H z| in FP32 (scaled V)
  unsigned long long best;  // bits of the best FP64 value so far (values are >= 0)
  unsigned long long counts;
};

// decide_fp32 for any K <= 8
__device__ __forceinline__ int enum_decide(float x, float y, int K, const EnumF32& tf) {
  const int BK = (K % 2 == 0) ? K / 2 : K;
  uint32_t s = 0;
#pragma unroll
  for (int m = 0; m < kMaxTcK; ++m)
    if (m < BK) s |= (fmaf(y, tf.bcos[m], -x * tf.bsin[m]) > 0.0f ? 1u : 0u) << m;
  if (K % 2 == 0) {
    const int c = __popc(s);
    return (s & 1u) ? c : (c == 0 ? 0 : K - c);
  }
  const uint32_t t = s & ~(s >> 1) & ((1u << (K - 1)) - 1u);
  return t ? __ffs(t) : 0;
}

// rank -> index set in the order of `unrank` (the largest index first, by
// bisection on the binomials)
__device__ inline void enum_unrank(unsigned long long rank, int N, int m, int* idx) {
  int hi = N;
  for (int pos = m; pos >= 1; --pos) {
    int lo = pos - 1, up = hi - 1;  // the largest c in [lo, up] with binom(c, pos) <= rank
    while (lo < up) {
      const int mid = (lo + up + 1) >> 1;
      if (binom(mid, pos) <= rank)
        lo = mid;
      else
        up = mid - 1;
    }
    idx[pos - 1] = lo;
    rank -= binom(lo, pos);
    hi = lo;
  }
}

// Upper bound of |V^H z|^2 over the candidates of vertex (index set I, sign)
// in the FP32 copy's scale, or INFINITY where FP32 cannot tell what the
// candidates are.  KT > 0: K known at compile time; RT: r known to be at most
// RT.  `unc` counts the coordinates whose FP32 decision is not certain, S is
// the sum with every coordinate's FP32 code.
template <int D, int KT, int RT>
__device__ __forceinline__ float enum_upper(const float2* __restrict__ V32, const float* __restrict__ rowb, int r,
                                            int K, const EnumF32& tf, int BK, const int* I, const float* cr,
                                            const float* ci, int sign, int unc, const float* sr, const float* si,
                                            float esum) {
  constexpr int M = 2 * D - 1;
  // the coordinates of I that touch a boundary here: their options
  int nb = 0, bi[M], bo[M][2], bc[M];
  int found = 0;
#pragma unroll
  for (int t = 0; t < M; ++t) {
    const int g = I[t] / BK;
    if (t > 0 && I[t - 1] / BK == g) continue;  // handled with its first row
    const bool dbl = t + 1 < M && I[t + 1] / BK == g;
    float x = 0.f, y = 0.f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float2 v = V32[g * r + j];
      x = fmaf(v.x, cr[j], fmaf(-v.y, ci[j], x));
      y = fmaf(v.x, ci[j], fmaf(v.y, cr[j], y));
    }
    if (sign < 0) {
      x = -x;
      y = -y;
    }
    const int k = KT > 0 ? decide_fp32<KT>(x, y, tf.bcos, tf.bsin) : enum_decide(x, y, K, tf);
    const int ka = k == 0 ? K - 1 : k - 1;
    const float pa = fmaf(y, tf.bcos[ka], -x * tf.bsin[ka]), pb = fmaf(y, tf.bcos[k], -x * tf.bsin[k]);
    const float b = rowb[g];
    const bool na = !(pa > b), nb_ = !(pb < -b);
    found += (na || nb_) ? 1 : 0;
    if (rowb[g] < 0.f) continue;  // a zero row: code 0, no contribution
    if (dbl) {
      bi[nb] = g;
      bo[nb][0] = k;
      bc[nb] = K;
      ++nb;
    } else if (na && nb_) {
      return INFINITY;  // w too small for FP32
    } else if (na || nb_) {
      bi[nb] = g;
      bo[nb][0] = k;
      bo[nb][1] = na ? ka : (k + 1 == K ? 0 : k + 1);
      bc[nb] = 2;
      ++nb;
    }
  }
  if (found != unc) return INFINITY;  // another coordinate is not certain
  int total = 1;
  for (int q = 0; q < nb; ++q) total *= bc[q];
  float best = 0.f;
  for (int ch = 0; ch < total; ++ch) {
    float tr[RT], ti[RT];
#pragma unroll
    for (int j = 0; j < RT; ++j) {
      tr[j] = sr[j];
      ti[j] = si[j];
    }
    int rem = ch;
    for (int q = 0; q < nb; ++q) {
      const int o = rem % bc[q];
      rem /= bc[q];
      const int k0 = bo[q][0], k1 = bc[q] == 2 ? bo[q][o] : o;
      if (k1 == k0) continue;
      const float dzr = tf.zr[k1] - tf.zr[k0], dzi = tf.zi[k1] - tf.zi[k0];
#pragma unroll
      for (int j = 0; j < RT; ++j) {
        if (j < r) {
          const float2 v = V32[bi[q] * r + j];
          tr[j] += v.x * dzr + v.y * dzi;
          ti[j] += v.x * dzi - v.y * dzr;
        }
      }
    }
    float f = 0.f;
#pragma unroll
    for (int j = 0; j < RT; ++j) f = fmaf(tr[j], tr[j], fmaf(ti[j], ti[j], f));
    best = fmaxf(best, f);
  }
  const float a = sqrtf(best) * 1.00001f + esum;
  return a * a * 1.00001f;
}

template <int D, int KT>
__global__ void __launch_bounds__(kEnumThreads) enum_kernel(const double2* __restrict__ V, int n, int r,
                                                            unsigned long long total, int per,
                                                            const __grid_constant__ EnumTables tb,
                                                            const __grid_constant__ EnumF32 tf,
                                                            const double* __restrict__ rown,
                                                            const float2* __restrict__ V32g,
                                                            const float* __restrict__ rowbg, EnumScan* scan,
                                                            EnumBest* __restrict__ block_best, int32_t* status) {
  constexpr int M = 2 * D - 1, NC = 2 * D;
  extern __shared__ __align__(16) uint8_t enum_smem[];
  float* lf = reinterpret_cast<float*>(enum_smem);                        // f_up of the vertices passed on
  int* lid = reinterpret_cast<int*>(lf + 2 * kEnumChunk);                 // 2 * set + (sign < 0)
  float2* V32 = reinterpret_cast<float2*>(lid + 2 * kEnumChunk);          // n x r
  float* rowb = reinterpret_cast<float*>(V32 + static_cast<size_t>(n) * r);  // bound of |p_m|'s error; -1: zero row
  __shared__ EnumBest sb[kEnumThreads];
  __shared__ int lcount;
  __shared__ float wmax[kEnumThreads / 32];
  for (int t = threadIdx.x; t < n * r; t += kEnumThreads) V32[t] = V32g[t];
  for (int t = threadIdx.x; t < n; t += kEnumThreads) rowb[t] = rowbg[t];
  const EnumV64 va{V, r, rown};
  const int K = KT > 0 ? KT : tb.K, BK = KT > 0 ? (KT % 2 == 0 ? KT / 2 : KT) : tb.BK;
  const int N = n * BK;
  const float esum = scan->esum;
  const double scale = scan->scale;
  // the best value so far in the FP32 copy's scale, rounded down
  auto best32 = [&]() {
    const double b = __longlong_as_double(static_cast<long long>(*reinterpret_cast<volatile unsigned long long*>(&scan->best)));
    return __double2float_rd(b * scale * scale * 0.99999999999);
  };
  EnumBest best;
  best.f = -1.0;
  best.level = 0;
  best.sign = 1;
  best.rank = 0;
  best.choice = 0;
  unsigned long long nfull = 0;
  const unsigned long long chunk_sets = static_cast<unsigned long long>(kEnumThreads) * per;
  const unsigned long long chunks = (total + chunk_sets - 1) / chunk_sets;
  for (unsigned long long chunk = blockIdx.x; chunk < chunks; chunk += gridDim.x) {
    if (threadIdx.x == 0) lcount = 0;
    __syncthreads();
    const unsigned long long c0 = chunk * chunk_sets;
    const unsigned long long r0 = c0 + static_cast<unsigned long long>(threadIdx.x) * per;
    const unsigned long long r1 = min(total, r0 + per);
    int I[M];
    if (r0 < r1) enum_unrank(r0, N, M, I);
    for (unsigned long long rk = r0; rk < r1; ++rk) {
      if (rk > r0) next_comb(N, M, I);
      if (!valid_set(I, M, BK)) continue;
      double H[M][NC], ct[NC];
#pragma unroll
      for (int t = 0; t < M; ++t) {
        const int i = I[t] / BK, mm = I[t] - i * BK;
        const double c = tb.rho_c[mm], s = tb.rho_s[mm];
#pragma unroll
        for (int j = 0; j < D; ++j) {
          const double vr = va.re(i, j), vi = va.im(i, j);
          H[t][j] = c * vi - s * vr;      // Im(rho V_ij)
          H[t][D + j] = c * vr + s * vi;  // Re(rho V_ij)
        }
      }
      if (!null_vector_fixed<M>(H, ct)) continue;
      ++nfull;
      float cr[D], ci[D];
#pragma unroll
      for (int j = 0; j < D; ++j) {
        cr[j] = static_cast<float>(ct[j]);
        ci[j] = static_cast<float>(ct[D + j]);
      }
      // both signs at once: -c has -w, so every boundary's side changes
      float sr[2][kEnumMaxD], si[2][kEnumMaxD];
      int unc[2] = {0, 0};
#pragma unroll
      for (int j = 0; j < kEnumMaxD; ++j) sr[0][j] = si[0][j] = sr[1][j] = si[1][j] = 0.f;
      for (int i = 0; i < n; ++i) {
        float vx[kEnumMaxD], vy[kEnumMaxD], x = 0.f, y = 0.f;
#pragma unroll
        for (int j = 0; j < kEnumMaxD; ++j) {
          vx[j] = vy[j] = 0.f;
          if (j < D || j < r) {
            const float2 v = V32[i * r + j];
            vx[j] = v.x;
            vy[j] = v.y;
          }
        }
#pragma unroll
        for (int j = 0; j < D; ++j) {
          x = fmaf(vx[j], cr[j], fmaf(-vy[j], ci[j], x));
          y = fmaf(vx[j], ci[j], fmaf(vy[j], cr[j], y));
        }
        const float b = rowb[i];
#pragma unroll
        for (int sgn = 0; sgn < 2; ++sgn) {
          const float xs = sgn ? -x : x, ys = sgn ? -y : y;
          const int k = KT > 0 ? decide_fp32<KT>(xs, ys, tf.bcos, tf.bsin) : enum_decide(xs, ys, K, tf);
          const int ka = k == 0 ? K - 1 : k - 1;
          const float pa = fmaf(ys, tf.bcos[ka], -xs * tf.bsin[ka]), pb = fmaf(ys, tf.bcos[k], -xs * tf.bsin[k]);
          unc[sgn] += (pa > b && pb < -b) ? 0 : 1;
          const float zr = tf.zr[k], zi = tf.zi[k];
#pragma unroll
          for (int j = 0; j < kEnumMaxD; ++j) {
            if (j < D || j < r) {
              sr[sgn][j] = fmaf(vx[j], zr, fmaf(vy[j], zi, sr[sgn][j]));
              si[sgn][j] = fmaf(vx[j], zi, fmaf(-vy[j], zr, si[sgn][j]));
            }
          }
        }
      }
      const float b32 = best32();
#pragma unroll
      for (int sgn = 0; sgn < 2; ++sgn) {
        const float up = enum_upper<D, KT, kEnumMaxD>(V32, rowb, r, K, tf, BK, I, cr, ci, sgn ? -1 : 1, unc[sgn],
                                                      sr[sgn], si[sgn], esum);
        if (!(up < b32)) {
          const int at = atomicAdd(&lcount, 1);
          lf[at] = up;
          lid[at] = 2 * static_cast<int>(rk - c0) + sgn;
        }
      }
    }
    __syncthreads();
    // FP64: the largest bound first, then what is still not below the best
    const int count = lcount;
    float mx = -1.f;
    for (int q = threadIdx.x; q < count; q += kEnumThreads) mx = fmaxf(mx, lf[q] < INFINITY ? lf[q] : 0.f);
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, q));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kEnumThreads / 32; ++q) mx = fmaxf(mx, wmax[q]);
    for (int pass = 0; pass < 2; ++pass) {
      const float b32 = best32();
      for (int q = threadIdx.x; q < count; q += kEnumThreads) {
        const float up = lf[q];
        const bool first = up == mx;
        if (pass == 0 ? !first : (first || up < b32)) continue;
        const unsigned long long rk = c0 + static_cast<unsigned>(lid[q] >> 1);
        int J[kEnumMaxRows];
        enum_unrank(rk, N, M, J);
        double H[kEnumMaxRows * 2 * kEnumMaxD], ct[2 * kEnumMaxD];
        build_rows(va, r, D, J, M, tb, H);
        if (!null_vector_fp64<kEnumMaxRows>(H, M, ct)) continue;
        EnumBest mine;
        mine.f = -1.0;
        eval_vertex(va, n, r, D, J, M, ct, (lid[q] & 1) ? -1 : 1, tb, mine, rk, -1, nullptr, nullptr, status);
        if (mine.f >= 0.0 && enum_better(mine, best)) best = mine;  // the list is not in rank order
        if (best.f >= 0.0)
          atomicMax(&scan->best, static_cast<unsigned long long>(__double_as_longlong(best.f)));
      }
      __syncthreads();
    }
  }
  sb[threadIdx.x] = best;
  if (nfull) atomicAdd(&scan->counts, nfull);
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      const EnumBest o = sb[threadIdx.x + h];
      if (enum_better(o, sb[threadIdx.x])) sb[threadIdx.x] = o;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) block_best[blockIdx.x] = sb[0];
}

// Squared row norms, the FP32 copy of V and its error bounds, and the input
// check; one block.
__global__ void __launch_bounds__(kEnumMaxN) enum_prep_kernel(const double2* __restrict__ V, int n, int r,
                                                              double* __restrict__ rown, float2* __restrict__ V32,
                                                              float* __restrict__ rowb, EnumScan* __restrict__ scan,
                                                              int32_t* status) {
  __shared__ double red[kEnumMaxN];
  const int i = threadIdx.x;
  double s = 0.0, mx = 0.0;
  bool finite = true;
  if (i < n) {
    for (int j = 0; j < r; ++j) {
      const double2 v = V[i * r + j];
      finite &= isfinite(v.x) && isfinite(v.y);
      s += v.x * v.x + v.y * v.y;
      mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
    }
    rown[i] = s;  // squared row norm
    if (!finite) dev_fail(status, LRQ_EINVAL);
  }
  red[i] = mx;
  __syncthreads();
  for (int h = kEnumMaxN / 2; h > 0; h >>= 1) {
    if (i < h) red[i] = fmax(red[i], red[i + h]);
    __syncthreads();
  }
  mx = red[0];
  __syncthreads();
  const int e = (mx > 0.0 && isfinite(mx)) ? ilogb(mx) : 0;
  const bool plain = e > -400 && e < 400;  // f and the scale's square stay in range
  const double scale = plain ? ldexp(1.0, -e) : 1.0;
  // rowb: 32 x 2^-24 sum |component| bounds the error of a boundary projection
  // ((2 r + 2) sqrt 2 + 6 roundings of terms below it at r <= 4) and, by a
  // factor above 1000, the 1e-9 |w| within which a coordinate is branched.
  // A row too small for FP32's range is never certain.
  double ab = 0.0;
  if (i < n) {
    for (int j = 0; j < r; ++j) {
      const double2 v = V[i * r + j];
      V32[i * r + j] = make_float2(static_cast<float>(v.x * scale), static_cast<float>(v.y * scale));
      ab += fabs(v.x) + fabs(v.y);
    }
    ab *= scale;
    rowb[i] = s == 0.0 ? -1.f : (ab > 1e-30 && finite ? static_cast<float>(ab) * (32.f * 5.9604645e-8f) : INFINITY);
  }
  // |V^H z| in FP32: each of the 2 r sums has at most 2 n + 24 roundings of
  // partial sums below sum_i |components of row i|
  red[i] = i < n ? ab : 0.0;
  __syncthreads();
  for (int h = kEnumMaxN / 2; h > 0; h >>= 1) {
    if (i < h) red[i] += red[i + h];
    __syncthreads();
  }
  if (i == 0) {
    scan->scale = scale;
    scan->esum = plain ? static_cast<float>(1.1 * sqrt(2.0) * red[0] * (2.0 * n + 24.0) * 5.9604645e-8) : INFINITY;
    scan->best = 0ull;
    scan->counts = 0ull;
  }
}

// One block: the best over all blocks of all levels, then its assignment.
// Lanes of the first warp take the coordinates in turn for the codes; the sum
// of component j is lane j's.
__global__ void __launch_bounds__(256) enum_final_kernel(const double2* __restrict__ V, int n, int r,
                                                         const __grid_constant__ EnumTables tb,
                                                         const double* __restrict__ rown,
                                                         const EnumBest* __restrict__ block_best, int nbest,
                                                         const EnumScan* __restrict__ scan,
                                                         uint8_t* __restrict__ z_out, double* __restrict__ f_out,
                                                         int64_t* __restrict__ n_sets_out) {
  __shared__ EnumBest sb[256];
  __shared__ uint8_t codes[kEnumMaxN];
  __shared__ uint8_t opts[kEnumMaxN];  // options of a coordinate, where more than one
  __shared__ double sct[2 * kEnumMaxD];
  __shared__ int sgrp[kEnumMaxRows];
  EnumBest best = block_best[0];
  for (int b = threadIdx.x; b < nbest; b += 256) {
    const EnumBest o = block_best[b];
    if (enum_better(o, best)) best = o;
  }
  sb[threadIdx.x] = best;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h && enum_better(sb[threadIdx.x + h], sb[threadIdx.x])) sb[threadIdx.x] = sb[threadIdx.x + h];
    __syncthreads();
  }
  best = sb[0];
  if (threadIdx.x == 0 && n_sets_out) *n_sets_out = static_cast<int64_t>(scan->counts);
  if (best.f < 0.0) {
    for (int i = threadIdx.x; i < n; i += 256) z_out[i] = 0;
    if (threadIdx.x == 0 && f_out) *f_out = -1.0;
    return;
  }
  const int d = best.level, m = 2 * d - 1;
  const EnumV64 va{V, r, rown};
  if (threadIdx.x == 0) {
    int I[kEnumMaxRows];
    enum_unrank(best.rank, n * tb.BK, m, I);
    double H[kEnumMaxRows * 2 * kEnumMaxD], ct[2 * kEnumMaxD];
    build_rows(va, r, d, I, m, tb, H);
    null_vector_fp64<kEnumMaxRows>(H, m, ct);
    for (int j = 0; j < 2 * d; ++j) sct[j] = best.sign * ct[j];
    for (int t = 0; t < m; ++t) sgrp[t] = I[t] / tb.BK;
  }
  __syncthreads();
  // the codes of eval_vertex; second options (a boundary's other side) are
  // the following code or, for the lower boundary, the code itself
  __shared__ uint8_t other[kEnumMaxN];
  for (int i = threadIdx.x; i < n; i += 256) {
    double x = 0.0, y = 0.0;
    for (int j = 0; j < d; ++j) {
      x += va.re(i, j) * sct[j] - va.im(i, j) * sct[d + j];
      y += va.re(i, j) * sct[d + j] + va.im(i, j) * sct[j];
    }
    int cnt_in = 0;
    for (int t = 0; t < m; ++t) cnt_in += (sgrp[t] == i);
    int opt[kMaxK];
    const int no = code_options(x, y, va.rownorm2(i), cnt_in >= 2, tb, opt);
    codes[i] = static_cast<uint8_t>(opt[0]);
    opts[i] = static_cast<uint8_t>(no);
    other[i] = static_cast<uint8_t>(no == 2 ? opt[1] : 0);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // the choice in mixed radix over the branched coordinates, in order; with
    // more than two options (all K) option q is code q
    unsigned long long rem = best.choice;
    for (int i = 0; i < n; ++i) {
      if (opts[i] <= 1) continue;
      const int q = static_cast<int>(rem % opts[i]);
      rem /= opts[i];
      if (q > 0) codes[i] = opts[i] == 2 ? other[i] : static_cast<uint8_t>(q);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += 256) z_out[i] = codes[i];
  if (threadIdx.x < 32) {
    const int j = threadIdx.x;
    double sr = 0.0, si = 0.0;
    if (j < r) {
      for (int i = 0; i < n; ++i) {
        const double vr = va.re(i, j), vi = va.im(i, j);
        sr += vr * tb.zr[codes[i]] + vi * tb.zi[codes[i]];
        si += vr * tb.zi[codes[i]] - vi * tb.zr[codes[i]];
      }
    }
    double f = sr * sr + si * si;
#pragma unroll
    for (int q = 4; q > 0; q >>= 1) f += __shfl_down_sync(0xffffffffu, f, q);
    if (j == 0 && f_out) *f_out = f;
  }
}

namespace {
struct EnumLayout {
  size_t off_rown, off_scan, off_v32, off_rowb, off_best, total;
};
EnumLayout enum_layout(int64_t n, int r) {
  EnumLayout l;
  size_t cur = 0;
  auto take = [&](size_t b) {
    const size_t o = cur;
    cur = align_up(cur + b, 256);
    return o;
  };
  l.off_rown = take(static_cast<size_t>(n) * sizeof(double));
  l.off_scan = take(sizeof(EnumScan));
  l.off_v32 = take(static_cast<size_t>(n) * r * sizeof(float2));
  l.off_rowb = take(static_cast<size_t>(n) * sizeof(float));
  l.off_best = take(static_cast<size_t>(kEnumMaxD) * kEnumBlocks * sizeof(EnumBest));  // per-block bests of every level
  l.total = cur;
  return l;
}
}  // namespace

size_t enum_workspace_bytes(int64_t n, int r) { return enum_layout(n, r).total; }

static unsigned long long host_binom(int nn, int k) {
  if (k < 0 || k > nn) return 0;
  long double b = 1;
  for (int t = 1; t <= k; ++t) b = b * (nn - k + t) / t;
  return b > 4.0e18L ? ~0ull : static_cast<unsigned long long>(b + 0.5L);
}

int enumerate_check(int64_t n, int r, int K, double budget) {
  if (n < 1) return fail(LRQ_EINVAL, "n must be >= 1");
  if (r < 1 || r > kMaxRank) return fail(LRQ_EINVAL, "r must be in [1, 8]");
  if (K < 2 || K > kMaxK) return fail(LRQ_EINVAL, "K must be in [2, 64]");
  if (n > kEnumMaxN) return fail(LRQ_EUNSUPPORTED, "lrq_enumerate supports n <= 512");
  if (r > kEnumMaxD) return fail(LRQ_EUNSUPPORTED, "lrq_enumerate supports r <= 4");
  if (K > kMaxTcK) return fail(LRQ_EUNSUPPORTED, "lrq_enumerate supports K <= 8");
  const double work = static_cast<double>(r) * std::pow(static_cast<double>(n), 2.0 * r + 1.0);
  if (work > (budget > 0.0 ? budget : kEnumDefaultBudget))
    return fail(LRQ_EUNSUPPORTED, "r * n^(2r+1) exceeds the enumeration budget");
  const int BK = (K % 2 == 0) ? K / 2 : K;
  const int N = static_cast<int>(n) * BK;
  for (int d = r; d >= 1; --d) {
    const unsigned long long t = host_binom(N, 2 * d - 1);
    // the device's incremental binomials multiply by at most N before dividing
    if (t == ~0ull || t > (1ull << 62) / static_cast<unsigned long long>(N))
      return fail(LRQ_EUNSUPPORTED, "too many index sets");
  }
  return LRQ_OK;
}

namespace {
struct EnumLaunch {
  const double2* V;
  int n, r;
  unsigned long long total;
  double* rown;
  EnumScan* scan;
  float2* V32;
  float* rowb;
  EnumBest* bests;
  int32_t* status;
  cudaStream_t st;
};

template <int D, int KT>
int enum_launch(const EnumLaunch& a, const EnumTables& tb, const EnumF32& tf, int* nbest) {
  // sets per thread: as many as leave two blocks per SM, at most
  // kEnumRanksPerThread (a thread unranks once per chunk)
  int per = 1;
  while (per < kEnumRanksPerThread &&
         a.total >= 2ull * per * kEnumThreads * 2 * static_cast<unsigned long long>(num_sms_current()))
    per *= 2;
  const unsigned long long sets = static_cast<unsigned long long>(kEnumThreads) * per;
  const int blocks = static_cast<int>(std::min<unsigned long long>((a.total + sets - 1) / sets, kEnumBlocks));
  const size_t smem = 2 * static_cast<size_t>(kEnumChunk) * 8 + static_cast<size_t>(a.n) * (a.r * 8 + 4);
  if (smem > 40 * 1024) {
    const int e = cuda_check(cudaFuncSetAttribute(enum_kernel<D, KT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  static_cast<int>(smem)),
                             "enumeration shared memory");
    if (e) return e;
  }
  enum_kernel<D, KT><<<blocks, kEnumThreads, smem, a.st>>>(a.V, a.n, a.r, a.total, per, tb, tf, a.rown, a.V32, a.rowb,
                                                           a.scan, a.bests, a.status);
  count_launch();
  *nbest += blocks;
  return cuda_check(cudaGetLastError(), "enum_kernel");
}

template <int D>
int enum_launch_k(const EnumLaunch& a, const EnumTables& tb, const EnumF32& tf, int* nbest) {
  switch (tb.K) {
    case 2: return enum_launch<D, 2>(a, tb, tf, nbest);
    case 3: return enum_launch<D, 3>(a, tb, tf, nbest);
    case 4: return enum_launch<D, 4>(a, tb, tf, nbest);
    default: return enum_launch<D, 0>(a, tb, tf, nbest);
  }
}

int enum_launch_level(const EnumLaunch& a, const EnumTables& tb, const EnumF32& tf, int d, int* nbest) {
  switch (d) {
    case 1: return enum_launch_k<1>(a, tb, tf, nbest);
    case 2: return enum_launch_k<2>(a, tb, tf, nbest);
    case 3: return enum_launch_k<3>(a, tb, tf, nbest);
    default: return enum_launch_k<4>(a, tb, tf, nbest);
  }
}
}  // namespace

int launch_enumerate(const double2* V, int64_t n, int r, int K, uint8_t* z_out, double* f_out, int64_t* n_sets_out,
                     void* ws, int32_t* status, cudaStream_t st) {
  const EnumTables tb = make_enum_tables(K);
  EnumF32 tf;
  for (int k = 0; k < kMaxTcK; ++k) {
    tf.zr[k] = static_cast<float>(tb.zr[k]);
    tf.zi[k] = static_cast<float>(tb.zi[k]);
    tf.bcos[k] = static_cast<float>(tb.bcos[k]);
    tf.bsin[k] = static_cast<float>(tb.bsin[k]);
  }
  const EnumLayout L = enum_layout(n, r);
  uint8_t* w = static_cast<uint8_t*>(ws);
  EnumLaunch a;
  a.V = V;
  a.n = static_cast<int>(n);
  a.r = r;
  a.rown = reinterpret_cast<double*>(w + L.off_rown);
  a.scan = reinterpret_cast<EnumScan*>(w + L.off_scan);
  a.V32 = reinterpret_cast<float2*>(w + L.off_v32);
  a.rowb = reinterpret_cast<float*>(w + L.off_rowb);
  a.status = status;
  a.st = st;
  EnumBest* bests = reinterpret_cast<EnumBest*>(w + L.off_best);
  enum_prep_kernel<<<1, kEnumMaxN, 0, st>>>(V, a.n, r, a.rown, a.V32, a.rowb, a.scan, status);
  count_launch();
  int nbest = 0, e;
  for (int d = r; d >= 1; --d) {
    a.total = host_binom(a.n * tb.BK, 2 * d - 1);
    if (a.total == 0) continue;  // enumerate_check bounded every level's count
    a.bests = bests + nbest;
    if ((e = enum_launch_level(a, tb, tf, d, &nbest))) return e;
  }
  enum_final_kernel<<<1, 256, 0, st>>>(V, a.n, r, tb, a.rown, bests, nbest, a.scan, z_out, f_out, n_sets_out);
  count_launch();
  return cuda_check(cudaGetLastError(), "enum_final_kernel");
}

}  // namespace lrq
