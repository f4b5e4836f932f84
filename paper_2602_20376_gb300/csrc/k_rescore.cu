// k_rescore.cu -- FP64-accurate re-scoring of selected candidates.
//
// For a selected direction c, recomputes w_i = V_i c, the decision rule of
// Sec. 3, Eq. 9 and f = ||V^H z||^2 (Sec. 4.2, Eq. 10) from the complex64 V
// and C taken exactly, so that the result equals the FP64 evaluation of the
// same candidate up to FP64 rounding.
//
// GB300 runs FP64 at about 1/64 of its FP32 rate, so the per-coordinate work
// avoids FP64 arithmetic while keeping FP64 accuracy:
//  * w is computed in FP32 together with a rigorous bound on its rounding
//    error; the FP32 decision is accepted only when both boundary lines of
//    the chosen sector are farther than that bound, which makes it equal to
//    the FP64 decision.  Otherwise w and the decision are recomputed in FP64
//    (rare: the angle must be within ~1e-6 of a boundary).
//  * conj(V_i) omega^k is accumulated in double-float form; a warp's (hi, lo)
//    pairs and the warps' sums are added by fixed trees.
//    For K in {2, 3, 4, 6} the roots of unity are omega^k = a + b tau with a, b in {-1, 0, 1}
//    (tau = i for K = 4, exp(i pi / 3) for K = 3 and 6), so the sums A = sum a
//    conj(V_i) and B = sum b conj(V_i) need no products: a sum's exact step
//    (two-sum, a or b folded into its FMAs) is 7 packed FP32 instructions for
//    both components, a warp's pairs are added in double-float, and V^H z = A +
//    tau B is formed in FP64 at the end.  Other alphabets multiply (exact products
//    by FMA residuals) and add a warp's pairs in three words.  Errors of f against
//    extended precision, n = 300 to 200003, the largest: K = 2, 3, 4, 6 6.9e-16
//    (1.4e-15 by products with FP64 sums over the warp), K = 5, 7, 8, 9, 16
//    1.7e-15 (as with FP64 over the warp; 5.1e-15 with double-float).
// The input check of V runs on the rows as they are staged.
#include <cuda_runtime.h>
#include <stdint.h>

#include "lrq_device.cuh"
#include "lrq_internal.h"
#include "score_f32x2.cuh"

namespace lrq {

constexpr int kRsThreads = 256;

struct RescoreTables {
  int K;
  float bcos[kMaxK], bsin[kMaxK];     // all K boundary lines, theta_m = pi(2m+1)/K
  double bcos64[kMaxK], bsin64[kMaxK];
  float zrh[kMaxK], zrl[kMaxK], zih[kMaxK], zil[kMaxK];  // omega^k as double-float
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// acc (hi, lo) += a*bh + a*bl + c*dh + c*dl with exact leading products
__device__ __forceinline__ void acc_dot2(float& hi, float& lo, float a, float bh, float bl, float c, float dh,
                                         float dl) {
  float p1 = a * bh;
  float e1 = fmaf(a, bh, -p1);
  float p2 = c * dh;
  float e2 = fmaf(c, dh, -p2);
  float s, e3;
  two_sum(p1, p2, s, e3);
  float small = fmaf(a, bl, fmaf(c, dl, (e1 + e2) + e3));
  float h2, e4;
  two_sum(hi, s, h2, e4);
  hi = h2;
  lo += e4 + small;
}

// (hi, lo) += v m, m a pair of multipliers in {-1, 0, 1}
__device__ __forceinline__ void acc_unit(f32x2& hi, f32x2& lo, f32x2 v, f32x2 m) { lo = add2(lo, add_unit(hi, v, m)); }

// omega^k = a + b tau
struct RootAB {
  signed char a[6], b[6];
};
template <int K>
__host__ __device__ constexpr RootAB root_ab() {
  if (K == 2) return RootAB{{1, -1}, {0, 0}};
  if (K == 3) return RootAB{{1, -1, 0}, {0, 1, -1}};
  if (K == 4) return RootAB{{1, 0, -1, 0}, {0, 1, 0, -1}};
  return RootAB{{1, 0, -1, -1, 0, 1}, {0, 1, 1, 0, -1, -1}};  // K = 6
}
template <int K>
struct RsLattice {
  static constexpr bool value = K == 2 || K == 3 || K == 4 || K == 6;
};

// Work split: a block takes kRsCpb candidates and one chunk of coordinates;
// the chunk's rows of V are staged through shared memory 256 at a time
// (component-major, so that the 32 lanes of a warp read 32 consecutive
// entries) and every warp evaluates its kRsCpw candidates on them, one row
// per lane.  V is thus read from memory once per kRsCpb candidates instead of
// once per candidate.  RM is the largest rank the instance handles (4 or 8):
// it sizes the per-thread accumulators.
// Bound: FP32 issue and pipe (K = 3, r = 4: about 100 instructions and 136
// pipe cycles an evaluation).  One candidate a warp, so that the registers leave
// three blocks an SM: with two a warp and two blocks the exact sums' chains of
// dependent instructions left 41% of the issue slots empty.  m = 64, n = 2^20,
// r = 4, K = 3: 477 us, 490 with two a warp; 673 with multiplied accumulation,
// FP32 scalars and a bound per evaluation (316 instructions).  m = 16, n = 3000:
// 7.3 us (11.1); r = 6, K = 8, m = 32, n = 50021: 33 us (45).
constexpr int kRsCpw = 1;                              // candidates per warp
constexpr int kRsCpb = kRsCpw * (kRsThreads / 32);     // candidates per block
constexpr int kRsTile = 256;                           // rows staged at a time
constexpr int kRsFlush = 256 * 32 / kRsTile;           // tiles between FP64 flushes (256 rows per lane)
static_assert(kRsCpw * 16 <= 32 && 2 * kMaxRank <= 16, "one lane per (candidate, component) total");

// (hi, lo) + (hi', lo') in double-float
__device__ __forceinline__ void add_pair(float& hi, float& lo, float h2, float l2) {
  const float t = hi + h2, b = t - hi;
  const float e = (hi - (t - b)) + (h2 - b) + (lo + l2);
  hi = t + e;
  lo = e - (hi - t);
}

// Sums N double-float values over the warp, halving the values at every step:
// lane l ends with the total of value l >> (5 - log2 N).  In double-float
// because FP64 instructions take a warp 16 cycles of its SM: sums in FP64 cost
// 10 us of the 21 that m = 16, n = 3000, r = 4, K = 3 took.
template <int N>
__device__ __forceinline__ void rs_warp_sums(float (&h)[N], float (&l)[N]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = N / 2, m = 16; m > 0; k >>= 1, m >>= 1) {
    if (k > 0) {
      const bool up = lane & m;
#pragma unroll
      for (int q = 0; q < (k > 0 ? k : 1); ++q) {
        const float gh = up ? h[q] : h[k + q], gl = up ? l[q] : l[k + q];
        h[q] = up ? h[k + q] : h[q];
        l[q] = up ? l[k + q] : l[q];
        add_pair(h[q], l[q], __shfl_xor_sync(0xffffffffu, gh, m), __shfl_xor_sync(0xffffffffu, gl, m));
      }
    } else {
      add_pair(h[0], l[0], __shfl_xor_sync(0xffffffffu, h[0], m), __shfl_xor_sync(0xffffffffu, l[0], m));
    }
  }
}

// (h, m, l) += (h', m', l') in three words: exact but for l's roundings.
__device__ __forceinline__ void add_triple(float& h, float& m, float& l, float h2, float m2, float l2) {
  float e, f, g, t;
  two_sum(h, h2, h, e);
  two_sum(m, m2, t, f);
  two_sum(t, e, m, g);
  l += l2 + (f + g);
}

// The same with a third word (l: 0 on entry), exact to 2^-60 or so: products' (hi,
// lo) pairs hold fewer bits than their FP64 sums, which double-float would lose
// (f off by three times as much at n = 300).  In FP64 it took 20 us of the 52 of
// r = 6, K = 8, m = 32, n = 50021 (a chunk is 220 rows there); 34 this way, 32 in
// double-float.
template <int N>
__device__ __forceinline__ void rs_warp_sums3(float (&h)[N], float (&m)[N], float (&l)[N]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = N / 2, x = 16; x > 0; k >>= 1, x >>= 1) {
    if (k > 0) {
      const bool up = lane & x;
#pragma unroll
      for (int q = 0; q < (k > 0 ? k : 1); ++q) {
        const float gh = up ? h[q] : h[k + q], gm = up ? m[q] : m[k + q], gl = up ? l[q] : l[k + q];
        h[q] = up ? h[k + q] : h[q];
        m[q] = up ? m[k + q] : m[q];
        l[q] = up ? l[k + q] : l[q];
        add_triple(h[q], m[q], l[q], __shfl_xor_sync(0xffffffffu, gh, x), __shfl_xor_sync(0xffffffffu, gm, x),
                   x == 16 ? 0.f : __shfl_xor_sync(0xffffffffu, gl, x));
      }
    } else {
      add_triple(h[0], m[0], l[0], __shfl_xor_sync(0xffffffffu, h[0], x), __shfl_xor_sync(0xffffffffu, m[0], x),
                 __shfl_xor_sync(0xffffffffu, l[0], x));
    }
  }
}

template <int K, int RM>
__global__ void __launch_bounds__(kRsThreads, RM <= 4 ? 3 : 2) rescore_partial_kernel(
    const float2* __restrict__ V, int64_t n, int r, const float2* __restrict__ C, int64_t S,
    const int64_t* __restrict__ idx, int m, int nchunk, int64_t rows_per_chunk, const __grid_constant__ RescoreTables tab,
    double* __restrict__ part, uint8_t* __restrict__ z_out, unsigned* __restrict__ done, int32_t* status) {
  constexpr bool LAT = RsLattice<K>::value;
  constexpr int NACC = LAT && K != 2 ? 2 : 1;  // A and B, or the sum itself
  constexpr int BKT = K == 0 ? 1 : ((K % 2 == 0) ? K / 2 : K);
  __shared__ float2 vs[RM][kRsTile];
  __shared__ float rowabs[kRsTile];
  __shared__ float2 cs[kRsCpb][RM];
  __shared__ float szrh[kMaxK], szrl[kMaxK], szih[kMaxK], szil[kMaxK];
  __shared__ float sbc[kMaxK], sbs[kMaxK];
  __shared__ double sbc64[kMaxK], sbs64[kMaxK];
  // per sign pattern: the code, and (lattice alphabets) {a, a, b, b}
  __shared__ float4 sab[LAT ? 1 << BKT : 1];
  __shared__ uint8_t scode[1 << BKT];
  const int Kr = (K > 0) ? K : tab.K;
  for (int k = threadIdx.x; k < Kr; k += blockDim.x) {
    sbc[k] = tab.bcos[k];
    sbs[k] = tab.bsin[k];
    sbc64[k] = tab.bcos64[k];
    sbs64[k] = tab.bsin64[k];
    szrh[k] = tab.zrh[k];
    szrl[k] = tab.zrl[k];
    szih[k] = tab.zih[k];
    szil[k] = tab.zil[k];
  }
  if constexpr (K > 0) {
    for (int t = threadIdx.x; t < 1 << BKT; t += blockDim.x) {
      const int k = decide_from_signs<K>(static_cast<uint32_t>(t));
      scode[t] = static_cast<uint8_t>(k);
      if constexpr (LAT) {
        constexpr RootAB ab = root_ab<K>();
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (q == k) {
            a = static_cast<float>(ab.a[q]);
            b = static_cast<float>(ab.b[q]);
          }
        sab[t] = make_float4(a, a, b, b);
      }
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.y;
  if (done && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *done = 0u;  // for rescore_sum_kernel
  const int tb = blockIdx.x * kRsCpb;  // first candidate position of the block
  for (int e = threadIdx.x; e < kRsCpb * RM; e += blockDim.x) {
    const int c = e / RM, j = e % RM;
    const int t = tb + c;
    float2 v = make_float2(0.f, 0.f);
    if (t < m && j < r) {
      const int64_t s = idx[t];
      if (s >= 0 && s < S) v = C[s * r + j];
    }
    cs[c][j] = v;
  }
  __syncthreads();

  // this warp's candidates
  int tc[kRsCpw];
  bool act[kRsCpw], ok[kRsCpw];
#pragma unroll
  for (int q = 0; q < kRsCpw; ++q) {
    tc[q] = tb + warp * kRsCpw + q;
    act[q] = tc[q] < m;
    const int64_t s = act[q] ? idx[tc[q]] : 0;
    ok[q] = act[q] && s >= 0 && s < S;
    if (act[q] && !ok[q] && lane == 0 && chunk == 0) dev_fail(status, LRQ_EINVAL);
  }
  float cr[kRsCpw][RM], ci[kRsCpw][RM], cb[kRsCpw];
#pragma unroll
  for (int q = 0; q < kRsCpw; ++q) {
    float mx = 0.f;
#pragma unroll
    for (int j = 0; j < RM; ++j) {
      const float2 c = cs[warp * kRsCpw + q][j];
      cr[q][j] = c.x;
      ci[q][j] = c.y;
      mx = fmaxf(mx, fabsf(c.x) + fabsf(c.y));
    }
    cb[q] = fp32_dir_bound(mx, r);  // the certificate's (score_f32x2.cuh)
  }
  f32x2 hi[kRsCpw][NACC][RM], lo[kRsCpw][NACC][RM];
#pragma unroll
  for (int q = 0; q < kRsCpw; ++q)
#pragma unroll
    for (int g = 0; g < NACC; ++g)
#pragma unroll
      for (int j = 0; j < RM; ++j) hi[q][g][j] = lo[q][g][j] = 0;
  // Every kRsFlush tiles (at most 256 rows per lane, which bounds the error
  // of the FP32 low parts) the lanes' (hi, lo) pairs are added over the warp
  // and the FP64 total of component j of candidate q is kept by lane q * 16 + j.
  double tot[NACC];
#pragma unroll
  for (int g = 0; g < NACC; ++g) tot[g] = 0.0;
  auto flush = [&]() {
#pragma unroll
    for (int g = 0; g < NACC; ++g) {
#pragma unroll
      for (int q = 0; q < kRsCpw; ++q) {
        float h[2 * RM], l[2 * RM];
#pragma unroll
        for (int j = 0; j < RM; ++j) {
          unpack2(hi[q][g][j], h[2 * j], h[2 * j + 1]);
          unpack2(lo[q][g][j], l[2 * j], l[2 * j + 1]);
          hi[q][g][j] = lo[q][g][j] = 0;
        }
        // value i ends in lane 32 / (2 RM) i; lane q * 16 + j takes it from there
        const int from = (32 / (2 * RM)) * (lane & 15) & 31;
        double mine;
        if constexpr (LAT) {
          rs_warp_sums(h, l);
          mine = static_cast<double>(__shfl_sync(0xffffffffu, h[0], from)) +
                 static_cast<double>(__shfl_sync(0xffffffffu, l[0], from));
        } else {
          float t[2 * RM];
#pragma unroll
          for (int j = 0; j < 2 * RM; ++j) t[j] = 0.f;
          rs_warp_sums3(h, l, t);
          mine = static_cast<double>(__shfl_sync(0xffffffffu, h[0], from)) +
                 (static_cast<double>(__shfl_sync(0xffffffffu, l[0], from)) +
                  static_cast<double>(__shfl_sync(0xffffffffu, t[0], from)));
        }
        if ((lane >> 4) == q) tot[g] += mine;
      }
    }
  };
  int tiles = 0;
  bool bad = false;

  const int64_t i0 = static_cast<int64_t>(chunk) * rows_per_chunk;
  const int64_t i1 = min(n, i0 + rows_per_chunk);
  for (int64_t ts = i0; ts < i1; ts += kRsTile) {
    if (tiles == kRsFlush) {
      flush();
      tiles = 0;
    }
    ++tiles;
    const int rows = static_cast<int>(min(static_cast<int64_t>(kRsTile), i1 - ts));
    __syncthreads();  // the previous tile has been read
    if (static_cast<int>(threadIdx.x) < rows) {
      const int row = threadIdx.x;  // kRsTile == kRsThreads: a row per thread
      float ab = 0.f;
#pragma unroll
      for (int j = 0; j < RM; ++j) {
        float2 v = make_float2(0.f, 0.f);
        if (j < r) v = V[(ts + row) * r + j];
        vs[j][row] = v;
        bad |= !isfinite(v.x) || !isfinite(v.y);
        ab += fabsf(v.x) + fabsf(v.y);
      }
      rowabs[row] = fp32_row_bound(ab);
    }
    __syncthreads();
    for (int ro = lane; ro < rows; ro += 32) {
      const int64_t i = ts + ro;
      float2 v[RM];
#pragma unroll
      for (int j = 0; j < RM; ++j) v[j] = vs[j][ro];
      const float ab = rowabs[ro];
#pragma unroll
      for (int q = 0; q < kRsCpw; ++q) {
        if (!act[q]) continue;
        float x = 0.f, y = 0.f;
#pragma unroll
        for (int j = 0; j < RM; ++j) {
          x = fmaf(v[j].x, cr[q][j], x);
          x = fmaf(-v[j].y, ci[q][j], x);
          y = fmaf(v[j].x, ci[q][j], y);
          y = fmaf(v[j].y, cr[q][j], y);
        }
        const float bound = fp32_proj_bound(ab, cb[q]);
        // certify: every boundary projection (K > 8, and odd K at second sight:
        // those of the sector's two boundaries) is farther from zero than its error
        bool sure;
        uint32_t s = 0;
        int k = 0;
        if constexpr (K > 0) {
          float pmin;
          s = sign_lines<K>(x, y, &pmin);
          sure = pmin > bound;
        } else {
          k = decide_fp32_generic(x, y, Kr);
          const int ma = (k == 0) ? Kr - 1 : k - 1;
          sure = fmaf(y, sbc[ma], -x * sbs[ma]) > bound && fmaf(y, sbc[k], -x * sbs[k]) < -bound;
        }
        if constexpr (K > 0 && K % 2 == 1) {
          // an odd alphabet's boundary is half of its line: w close to the other
          // half is certain by its sector's own two boundaries
          if (!sure) {
            const int kk = scode[s], ma = kk == 0 ? K - 1 : kk - 1;
            sure = fmaf(y, sbc[ma], -x * sbs[ma]) > bound && fmaf(y, sbc[kk], -x * sbs[kk]) < -bound;
          }
        }
        if (!sure) {
          double xd = 0.0, yd = 0.0;
#pragma unroll
          for (int j = 0; j < RM; ++j) {
            xd = fma(static_cast<double>(v[j].x), static_cast<double>(cr[q][j]), xd);
            xd = fma(-static_cast<double>(v[j].y), static_cast<double>(ci[q][j]), xd);
            yd = fma(static_cast<double>(v[j].x), static_cast<double>(ci[q][j]), yd);
            yd = fma(static_cast<double>(v[j].y), static_cast<double>(cr[q][j]), yd);
          }
          k = decide_fp64(xd, yd, Kr, sbc64, sbs64);
          if constexpr (K > 0) s = pattern_of<K>(k);
        }
        if constexpr (K > 0) {
          if (!LAT || z_out) k = scode[s];
        }
        if (z_out && ok[q]) z_out[static_cast<int64_t>(tc[q]) * n + i] = static_cast<uint8_t>(k);
        if constexpr (LAT) {
          const ulonglong2 ab2 = reinterpret_cast<const ulonglong2*>(sab)[s];
#pragma unroll
          for (int j = 0; j < RM; ++j) {
            if (j < r) {
              const f32x2 vv = pack2(v[j].x, -v[j].y);  // conj(V_ij)
              acc_unit(hi[q][0][j], lo[q][0][j], vv, ab2.x);
              if constexpr (NACC == 2) acc_unit(hi[q][1][j], lo[q][1][j], vv, ab2.y);
            }
          }
        } else {
          const float zrh = szrh[k], zrl = szrl[k], zih = szih[k], zil = szil[k];
#pragma unroll
          for (int j = 0; j < RM; ++j) {
            if (j < r) {
              // Re(conj(V) z) = vr zr + vi zi ; Im(conj(V) z) = vr zi - vi zr
              float hr, hm, lr, lm;
              unpack2(hi[q][0][j], hr, hm);
              unpack2(lo[q][0][j], lr, lm);
              acc_dot2(hr, lr, v[j].x, zrh, zrl, v[j].y, zih, zil);
              acc_dot2(hm, lm, v[j].x, zih, zil, -v[j].y, zrh, zrl);
              hi[q][0][j] = pack2(hr, hm);
              lo[q][0][j] = pack2(lr, lm);
            }
          }
        }
      }
    }
  }
  flush();
  if (bad && blockIdx.x == 0) dev_fail(status, LRQ_EINVAL);
  {
    const int q = lane >> 4, j = lane & 15;
    double out = tot[0];
    if constexpr (NACC == 2) {
      // + tau B: re -= / += by the partner component
      const double other = __shfl_xor_sync(0xffffffffu, tot[1], 1);
      const double tr = K == 4 ? 0.0 : 0.5, ti = K == 4 ? 1.0 : 0.86602540378443864676;
      out += tr * tot[1] + ((j & 1) ? ti : -ti) * other;
    }
    if (q < kRsCpw && j < 2 * r && act[q < kRsCpw ? q : 0]) part[(static_cast<int64_t>(tc[q]) * nchunk + chunk) * (2 * kMaxRank) + j] = out;
  }
}

// f of every candidate, a block each, and the best of the m (largest f, ties to
// the earlier position) by the last block to finish.  What bounds it is FP64: a
// warp-wide FP64 add holds an SM's FP64 unit (two lanes wide) for 16 cycles.  So
// candidates spread over the SMs, a lane holds one component (16 lanes a chunk,
// eight chunks at a time: coalesced) and only 12 additions follow the chunk
// sums; all orders are fixed.  One block of eight warps took 77.6 us at m = 64,
// 107.5 us at m = 164; a warp per candidate, each lane all components, 4.6-12 us
// and 2.6 us for the best in a launch of its own; now 5-9.
constexpr int kRsSumThreads = 128;

__global__ void __launch_bounds__(kRsSumThreads) rescore_sum_kernel(const double* __restrict__ part, int nchunk, int r,
                                                                    const int64_t* __restrict__ idx, int64_t S,
                                                                    double* f_out, unsigned* done, int64_t* best_out,
                                                                    double* best_f_out) {
  constexpr int NG = kRsSumThreads / 16;  // chunks at a time
  __shared__ double red[kRsSumThreads / 32][16];
  __shared__ bool last;
  __shared__ double bf[kRsSumThreads / 32];
  __shared__ int bt[kRsSumThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = threadIdx.x & 15, t = blockIdx.x;
  double a = 0.0;
  if (j < 2 * r) {
    const double* p = part + static_cast<int64_t>(t) * nchunk * (2 * kMaxRank) + j;
#pragma unroll 4
    for (int c = threadIdx.x >> 4; c < nchunk; c += NG) a += p[static_cast<int64_t>(c) * (2 * kMaxRank)];
  }
  a += __shfl_xor_sync(0xffffffffu, a, 16);
  if (lane < 16) red[warp][lane] = a;
  __syncthreads();
  if (warp == 0) {
    double v = red[0][j];
#pragma unroll
    for (int w = 1; w < kRsSumThreads / 32; ++w) v += red[w][j];
    double f = v * v;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) f += __shfl_xor_sync(0xffffffffu, f, off);
    if (lane == 0) {
      const int64_t s = idx[t];
      f_out[t] = (s < 0 || s >= S) ? -1.0 : f;
      last = false;
      if (done) {
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
        __threadfence();
      }
    }
  }
  __syncthreads();
  if (!last) return;
  const int m = gridDim.x;
  double my_best = -1.0;
  int my_t = 0x7fffffff;
  auto take = [&](double f, int at) {
    if (f > my_best || (f == my_best && at < my_t)) {
      my_best = f;
      my_t = at;
    }
  };
  for (int q = threadIdx.x; q < m; q += kRsSumThreads) take(__ldcg(f_out + q), q);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double f = __shfl_xor_sync(0xffffffffu, my_best, off);
    take(f, __shfl_xor_sync(0xffffffffu, my_t, off));
  }
  if (lane == 0) {
    bf[warp] = my_best;
    bt[warp] = my_t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < kRsSumThreads / 32; ++w) take(bf[w], bt[w]);
    if (best_out) *best_out = my_t < m ? idx[my_t] : -1;
    if (best_f_out) *best_f_out = my_best;
  }
}

int rescore_blocks_x(int m) { return (m + kRsCpb - 1) / kRsCpb; }

int launch_rescore(const RescorePlan& p, const Alphabet& a, const float2* V, const float2* C, int64_t S,
                   const int64_t* idx, double* part, double* f_out, uint8_t* z_out, int64_t* best_out,
                   double* best_f_out, int32_t* status, cudaStream_t st) {
  RescoreTables tab;
  tab.K = a.K;
  for (int k = 0; k < kMaxK; ++k) {
    bool in = k < a.K;
    // all K boundary lines (not only the B_K distinct ones)
    double th = kPi * (2.0 * k + 1.0) / a.K;
    double c = in ? cos(th) : 0.0, s = in ? sin(th) : 0.0;
    if (fabs(c) < 1e-15) c = 0.0;
    if (fabs(s) < 1e-15) s = 0.0;
    tab.bcos64[k] = c;
    tab.bsin64[k] = s;
    tab.bcos[k] = static_cast<float>(c);
    tab.bsin[k] = static_cast<float>(s);
    double zr = in ? a.zr64[k] : 0.0, zi = in ? a.zi64[k] : 0.0;
    tab.zrh[k] = static_cast<float>(zr);
    tab.zrl[k] = static_cast<float>(zr - static_cast<double>(tab.zrh[k]));
    tab.zih[k] = static_cast<float>(zi);
    tab.zil[k] = static_cast<float>(zi - static_cast<double>(tab.zih[k]));
  }
  dim3 grid(static_cast<unsigned>(rescore_blocks_x(p.m)), static_cast<unsigned>(p.nchunk));
  // counts the finished candidates, in an output's eight bytes until its value is written
  unsigned* const done = best_out ? reinterpret_cast<unsigned*>(best_out) : reinterpret_cast<unsigned*>(best_f_out);
#define LRQ_RS_LAUNCH(KK, RR)                                                                                \
  rescore_partial_kernel<KK, RR><<<grid, kRsThreads, 0, st>>>(V, p.n, p.r, C, S, idx, p.m, p.nchunk,         \
                                                              p.rows_per_chunk, tab, part, z_out, done, status)
#define LRQ_RS_CASE(KK)             \
  case KK:                          \
    if (p.r <= 4)                   \
      LRQ_RS_LAUNCH(KK, 4);         \
    else                            \
      LRQ_RS_LAUNCH(KK, kMaxRank);  \
    break;
  switch (a.K <= 8 ? a.K : 0) {
    LRQ_RS_CASE(2)
    LRQ_RS_CASE(3)
    LRQ_RS_CASE(4)
    LRQ_RS_CASE(5)
    LRQ_RS_CASE(6)
    LRQ_RS_CASE(7)
    LRQ_RS_CASE(8)
    LRQ_RS_CASE(0)
  }
#undef LRQ_RS_CASE
#undef LRQ_RS_LAUNCH
  count_launch();
  int e = cuda_check(cudaGetLastError(), "rescore_partial_kernel");
  if (e) return e;
  rescore_sum_kernel<<<static_cast<unsigned>(p.m), kRsSumThreads, 0, st>>>(part, p.nchunk, p.r, idx, S, f_out, done,
                                                                           best_out, best_f_out);
  count_launch();
  return cuda_check(cudaGetLastError(), "rescore_sum_kernel");
}

}  // namespace lrq
