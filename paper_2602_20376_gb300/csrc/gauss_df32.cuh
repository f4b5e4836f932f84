// gauss_df32.cuh -- Box-Muller in double-float arithmetic: the draws of
// sphere_component (lrq_device.cuh) on the FP32 units.
//
// GB300 runs FP64 at 1/64 of its FP32 rate and a Box-Muller pair takes about
// 120 FP64 instructions (log, sqrt, sincospi).  Here a value is an unevaluated
// sum hi + lo of two FP32 numbers (Dekker; products split exactly by FMA,
// sums by Knuth's two-sum), and the functions are table-driven reductions
// (Tang) with short Taylor polynomials whose leading terms are double-float:
//   -ln u     u = 2^-k f, f in [0.707, 1.414); 1 / c for the nearest c = i/256
//             to f, s = f / c - 1 formed exactly for c = 1, so that the result
//             keeps its relative accuracy as u -> 1; ln(1 + s) to s^6
//   sin, cos  of 2 pi u: the nearest of 256 angles (its sine and cosine as
//             double-floats), the remainder's sine to b^5 and cosine to b^4
// The uniforms' 54-bit integers 2 x + 1 (u = (2 x + 1) 2^-54) are taken apart
// exactly.  Errors against extended precision over 2 * 10^7 draws (with many
// near 0 and 1): -ln u below 2^-39 relative, sine and cosine below 2^-45
// absolute.  A direction's component that lies this close to the middle of two
// FP32 numbers (about one in 5000) is drawn again in FP64, so that every
// component is the rounded 64-bit one.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "lrq_device.cuh"

#define LRQ_HD __host__ __device__ __forceinline__

namespace lrq {

struct df32 {
  float h, l;
};

#ifdef __CUDA_ARCH__
LRQ_HD float df_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
LRQ_HD float df_add(float a, float b) { return __fadd_rn(a, b); }
LRQ_HD float df_mul(float a, float b) { return __fmul_rn(a, b); }
#else
LRQ_HD float df_fma(float a, float b, float c) { return fmaf(a, b, c); }
LRQ_HD float df_add(float a, float b) { return a + b; }
LRQ_HD float df_mul(float a, float b) { return a * b; }
#endif
LRQ_HD float df_sub(float a, float b) { return df_add(a, -b); }

LRQ_HD df32 df_two_sum(float a, float b) {
  const float s = df_add(a, b), bb = df_sub(s, a);
  return df32{s, df_add(df_sub(a, df_sub(s, bb)), df_sub(b, bb))};
}
LRQ_HD df32 df_fast_sum(float a, float b) {  // |a| >= |b| or a = 0
  const float s = df_add(a, b);
  return df32{s, df_sub(b, df_sub(s, a))};
}
LRQ_HD df32 df_prod(float a, float b) {
  const float p = df_mul(a, b);
  return df32{p, df_fma(a, b, -p)};
}
LRQ_HD df32 df_sum(df32 a, df32 b) {
  const df32 s = df_two_sum(a.h, b.h);
  return df_fast_sum(s.h, df_add(s.l, df_add(a.l, b.l)));
}
LRQ_HD df32 df_times(df32 a, df32 b) {
  const df32 p = df_prod(a.h, b.h);
  return df_fast_sum(p.h, df_add(p.l, df_fma(a.h, b.l, df_mul(a.l, b.h))));
}

// Tables, evaluated at compile time in double: for c = i / 256, i = 181..362
// (index i - 181), {fl(1/c), -ln(fl(1/c)) as hi, lo}; for j = 0..255 sine and
// cosine of 2 pi j / 256 as {sin hi, sin lo, cos hi, cos lo}.
struct GaussTables {
  float rc[182][4];
  float sc[256][4];
};

constexpr double gauss_ln(double x) {  // 2 atanh((x - 1) / (x + 1)), x in [0.7, 1.42]
  const double t = (x - 1.0) / (x + 1.0), t2 = t * t;
  double s = 0.0;
  for (int k = 39; k >= 1; k -= 2) s = s * t2 + 1.0 / k;
  return 2.0 * t * s;
}
constexpr double gauss_sin(double x) {  // Taylor, |x| <= pi / 4
  double s = 0.0;
  for (int k = 21; k >= 3; k -= 2) s = (1.0 + s) * (-x * x / (k * (k - 1.0)));
  return x * (1.0 + s);
}
constexpr double gauss_cos(double x) {
  double s = 0.0;
  for (int k = 20; k >= 2; k -= 2) s = (1.0 + s) * (-x * x / (k * (k - 1.0)));
  return 1.0 + s;
}
constexpr GaussTables make_gauss_tables() {
  GaussTables t{};
  for (int i = 0; i < 182; ++i) {
    const float rc = static_cast<float>(256.0 / (i + 181));
    const double l = -gauss_ln(static_cast<double>(rc));
    t.rc[i][0] = rc;
    t.rc[i][1] = static_cast<float>(l);
    t.rc[i][2] = static_cast<float>(l - static_cast<double>(t.rc[i][1]));
  }
  for (int j = 0; j < 256; ++j) {
    const int q = ((j + 32) / 64) % 4, d = j - ((j + 32) / 64) * 64;  // quadrant axis and offset, |d| <= 32
    const double x = kPi * d / 128.0, sn = gauss_sin(x), cs = gauss_cos(x);
    const double a = q == 0 ? sn : (q == 1 ? cs : (q == 2 ? -sn : -cs));
    const double b = q == 0 ? cs : (q == 1 ? -sn : (q == 2 ? -cs : sn));
    t.sc[j][0] = static_cast<float>(a);
    t.sc[j][1] = static_cast<float>(a - static_cast<double>(t.sc[j][0]));
    t.sc[j][2] = static_cast<float>(b);
    t.sc[j][3] = static_cast<float>(b - static_cast<double>(t.sc[j][2]));
  }
  return t;
}
static __device__ const GaussTables g_gauss = make_gauss_tables();

// the device's copy, read 16 bytes at a time
struct GaussTab {
  __device__ float4 log_row(int i) const { return __ldg(reinterpret_cast<const float4*>(g_gauss.rc[i])); }
  __device__ float4 sc_row(int j) const { return __ldg(reinterpret_cast<const float4*>(g_gauss.sc[j])); }
};

// A 54-bit odd integer as the exact sum of three floats (18 bits each).
LRQ_HD void df_split54(uint64_t U, float* a, float* b, float* c) {
  *a = static_cast<float>(static_cast<uint32_t>(U >> 36)) * 68719476736.0f;         // 2^36
  *b = static_cast<float>(static_cast<uint32_t>((U >> 18) & 0x3ffffu)) * 262144.0f;  // 2^18
  *c = static_cast<float>(static_cast<uint32_t>(U & 0x3ffffu));
}

// k ln 2 - ln f for f = a + b + c in [0.707, 1.414], |b| below 2^-17, |c|
// below 2^-35 or so (a - 1 then is exact)
template <class Tab>
LRQ_HD df32 df_neg_log_core(float a, float b, float c, int k, const Tab& tab) {
  const float f = df_add(a, b);
  const int i = static_cast<int>(f * 256.0f + 0.5f);  // 181 .. 362
  const float4 row = tab.log_row(i - 181);
  const float rc = row.x;
  const df32 lc{row.y, row.z};
  // s = f rc - 1: a rc - 1 is exact up to the product's remainder
  const df32 pa = df_prod(a, rc), pb = df_prod(b, rc);
  const df32 t = df_two_sum(df_sub(pa.h, 1.0f), pb.h);
  const df32 s = df_fast_sum(t.h, df_add(t.l, df_add(pa.l, df_add(pb.l, df_mul(c, rc)))));
  // ln(1 + s) = s - s^2/2 + s^3 (1/3 - s/4 + s^2/5 - s^3/6)
  const float q = df_fma(s.h, df_fma(s.h, df_fma(s.h, -1.0f / 6.0f, 0.2f), -0.25f), 1.0f / 3.0f);
  df32 s2 = df_prod(s.h, s.h);
  s2.l = df_fma(2.0f * s.h, s.l, s2.l);
  const float tail = df_mul(df_mul(s2.h, s.h), q);
  df32 ln = df_fast_sum(s.h, -0.5f * s2.h);
  ln.l = df_add(ln.l, df_add(s.l, df_fma(-0.5f, s2.l, tail)));
  // k ln 2 - lc - ln; ln 2 in an 18-bit head (exact times k) and a tail
  const float kf = static_cast<float>(k);
  const df32 k2 = df_fast_sum(df_mul(kf, 0x1.62e4p-1f), df_mul(kf, 0x1.7f7d1cp-20f));
  const df32 base = df_sum(df32{k2.h, df_add(k2.l, df_mul(kf, 0x1.ef357ap-45f))}, df32{-lc.h, -lc.l});
  return df_sum(base, df32{-ln.h, -ln.l});
}

// U = m 2^-shift with m's leading bit at 2^53 (U odd, below 2^54)
LRQ_HD uint64_t df_normalise(uint64_t U, int* shift) {
#ifdef __CUDA_ARCH__
  *shift = __clzll(static_cast<long long>(U)) - 10;
#else
  *shift = __builtin_clzll(U) - 10;
#endif
  return U << *shift;
}

// -ln(U 2^-54) for odd U < 2^54
template <class Tab>
LRQ_HD df32 df_neg_log(uint64_t U, const Tab& tab) {
  // f = U 2^-(54 - k) in [0.707, 1.414): by the position of the leading bit
  int shift;
  const uint64_t m = df_normalise(U, &shift);
  const bool up = m >= 12737979836874752ull;  // 1.41421356 2^53: above sqrt(2), f = m / 2^54
  float a, b, c;
  df_split54(m, &a, &b, &c);
  const float sc = up ? 0x1p-54f : 0x1p-53f;
  return df_neg_log_core(a * sc, b * sc, c * sc, up ? shift : shift + 1, tab);
}

// -ln of the product of three uniforms U 2^-54 (2^-44 of the product's
// rounding on top)
template <class Tab>
LRQ_HD df32 df_neg_log3(uint64_t U1, uint64_t U2, uint64_t U3, const Tab& tab) {
  int k = 3, sh;  // u = m 2^-53 2^-(shift + 1)
  df32 p{1.f, 0.f};
  const uint64_t U[3] = {U1, U2, U3};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const uint64_t m = df_normalise(U[q], &sh);
    k += sh;
    float a, b, c;
    df_split54(m, &a, &b, &c);
    df32 t = df_fast_sum(a * 0x1p-53f, b * 0x1p-53f);
    t = df_fast_sum(t.h, df_add(t.l, c * 0x1p-53f));
    p = q == 0 ? t : df_times(p, t);
  }
  // p in [1, 8)
  const int e = p.h >= 5.6568542f ? 3 : (p.h >= 2.8284271f ? 2 : (p.h >= 1.4142135f ? 1 : 0));
  const float sc = e == 3 ? 0.125f : (e == 2 ? 0.25f : (e == 1 ? 0.5f : 1.0f));
  return df_neg_log_core(p.h * sc, p.l * sc, 0.f, k - e, tab);
}

// cos and sin of 2 pi U 2^-54
template <class Tab>
LRQ_HD void df_sincos(uint64_t U, const Tab& tab, df32* sn, df32* cs) {
  const uint64_t j = (U + (1ull << 45)) >> 46;
  const int64_t d = static_cast<int64_t>(U) - static_cast<int64_t>(j << 46);  // |d| <= 2^45
  const float d1 = static_cast<float>(static_cast<int32_t>(d >> 23)) * 8388608.0f;
  const float d0 = static_cast<float>(static_cast<int32_t>(d & 0x7fffff));
  const df32 dd = df_fast_sum(d1, d0);
  // b = 2 pi d 2^-54
  const df32 b = df_times(df32{dd.h * 0x1p-54f, dd.l * 0x1p-54f}, df32{0x1.921fb6p+2f, -0x1.777a5cp-23f});
  df32 b2 = df_prod(b.h, b.h);
  b2.l = df_fma(2.0f * b.h, b.l, b2.l);
  // sin b = b - b b^2 / 6 + b^5 / 120, cos b - 1 = -b^2 / 2 + b^4 / 24
  const float b4 = df_mul(b2.h, b2.h);
  const df32 t = df_prod(b2.h, df_mul(b.h, -1.0f / 6.0f));
  // -b^3/6 with the rounding of b / 6 put back: b b^2 (-1/6) exactly is
  // b2.h (b.h / -6 + r), r = (-b.h - 6 fl(b.h / -6)) / 6
  const float b6 = df_mul(b.h, -1.0f / 6.0f);
  const float r6 = df_mul(df_fma(-6.0f, b6, -b.h), 1.0f / 6.0f);
  df32 sb = df_fast_sum(b.h, t.h);
  float lo = df_add(t.l, df_mul(b2.h, r6));
  lo = df_add(lo, df_fma(b2.l, b6, df_mul(b2.h, df_mul(b.l, -0.5f))));
  lo = df_fma(df_mul(b4, b.h), 1.0f / 120.0f, lo);
  sb.l = df_add(sb.l, df_add(b.l, lo));
  const df32 cm{-0.5f * b2.h, df_fma(b4, 1.0f / 24.0f, -0.5f * b2.l)};
  const int jj = static_cast<int>(j & 255u);
  const float4 row = tab.sc_row(jj);
  const df32 sA{row.x, row.y}, cA{row.z, row.w};
  auto mul = [](df32 x, df32 y) {  // product, not renormalised
    const df32 p = df_prod(x.h, y.h);
    return df32{p.h, df_add(p.l, df_fma(x.h, y.l, df_mul(x.l, y.h)))};
  };
  auto plus = [](df32 x, df32 y, df32 z) {  // x + (y + z), |z| below |y| or so
    const df32 u = df_two_sum(y.h, z.h);
    const df32 v = df_two_sum(x.h, u.h);
    return df_fast_sum(v.h, df_add(v.l, df_add(df_add(u.l, df_add(y.l, z.l)), x.l)));
  };
  const df32 p1 = mul(cA, sb), p2 = mul(sA, cm), p3 = mul(sA, sb), p4 = mul(cA, cm);
  *sn = plus(sA, p1, p2);
  *cs = plus(cA, df32{-p3.h, -p3.l}, p4);
}

// sqrt of a non-negative double-float
LRQ_HD df32 df_sqrt(df32 x) {
#ifdef __CUDA_ARCH__
  const float r = __fsqrt_rn(x.h);
#else
  const float r = sqrtf(x.h);
#endif
  const float e = df_add(df_fma(-r, r, x.h), x.l);
  return df_fast_sum(r, r > 0.0f ? e / (2.0f * r) : 0.0f);
}

// 1 / x
LRQ_HD df32 df_recip(df32 x) {
  const float r = 1.0f / x.h;
  const float e = df_fma(-r, x.l, df_fma(-r, x.h, 1.0f));
  return df_fast_sum(r, df_mul(r, e));
}

// Whether rounding h + l (h the nearest FP32 number) may depend on an error of err.
__device__ __forceinline__ bool df_near_midpoint(df32 x, float err) {
  const uint32_t b = __float_as_uint(x.h) & 0x7fffffffu;
  if ((b & 0x7fffffu) == 0u || b < (24u << 23)) return true;  // a power of two (half the spacing below), tiny
  const float half = __uint_as_float((b & 0x7f800000u) - (24u << 23));
  return half - fabsf(x.l) <= err;
}
// The same for a direction's component: 2^-37 of it plus 2^-43 are above its error
// (g within 2^-38, sine and cosine 2^-45).
__device__ __forceinline__ bool df_near_midpoint(df32 x) {
  return df_near_midpoint(x, fmaf(fabsf(x.h), 0x1p-37f, 0x1p-43f));
}

// The directions of a block of 256 threads (lrq_sample_directions' draws): a
// thread per component, 256 / r candidates a block, ||Z||^2 = sum_j -ln u1_j
// exchanged through shared memory.  A candidate with a component near a midpoint
// is drawn again in FP64 by its r threads side by side (one thread doing it alone
// for its component took 5.2 ms for 300000 directions of r = 64, 0.8 so, and 14.7
// us for 2^14 of r = 4, 6.8 so).  s_first: the block's first candidate; every
// thread of the block calls it.
constexpr int kSphereThreads = 256;
__host__ __device__ inline int sphere_per_block(int r) { return kSphereThreads / r; }

__device__ __forceinline__ void sphere_block(uint64_t seed, int64_t s_first, int64_t S, int r, float2* __restrict__ C) {
  __shared__ df32 nl[kSphereThreads];
  __shared__ double nd[kSphereThreads];
  __shared__ uint8_t again[kSphereThreads];  // by candidate
  const int per = sphere_per_block(r);
  const int c = threadIdx.x / r, j = threadIdx.x - c * r;
  const int64_t s = s_first + c;
  const bool act = c < per && s < S;
  uint64_t U2 = 1;
  df32 L{1.f, 0.f};
  if (act) {
    const PhiloxOut o = philox4x32_10(static_cast<uint32_t>(s), static_cast<uint32_t>(static_cast<uint64_t>(s) >> 32),
                                      static_cast<uint32_t>(j), 0u, static_cast<uint32_t>(seed),
                                      static_cast<uint32_t>(seed >> 32));
    // the uniforms' 2 x + 1, x the top 53 bits of the two words
    const uint64_t U1 = ((((static_cast<uint64_t>(o.w[0]) << 32) | o.w[1]) >> 11) << 1) | 1ull;
    U2 = ((((static_cast<uint64_t>(o.w[2]) << 32) | o.w[3]) >> 11) << 1) | 1ull;
    L = df_neg_log(U1, GaussTab());
  }
  nl[threadIdx.x] = L;
  again[threadIdx.x] = 0;
  __syncthreads();
  float2 out = make_float2(0.f, 0.f);
  bool unsure = false;
  if (act) {
    df32 N = nl[c * r];
    for (int k = 1; k < r; ++k) N = df_sum(N, nl[c * r + k]);
    df32 sn, cs;
    df_sincos(U2, GaussTab(), &sn, &cs);
    const df32 g = df_times(df_sqrt(L), df_recip(df_sqrt(N)));
    const df32 re = df_times(g, cs), im = df_times(g, sn);
    out = make_float2(re.h, im.h);
    unsure = df_near_midpoint(re) || df_near_midpoint(im);
    if (unsure) again[c] = 1;
  }
  if (__syncthreads_or(unsure)) {
    double a = 0.0, b = 0.0;
    const bool mine = act && again[c];
    if (mine) {
      sphere_component(seed, s, j, &a, &b);
      nd[threadIdx.x] = a * a + b * b;
    }
    __syncthreads();
    if (mine && unsure) {
      double nrm2 = 0.0;
      for (int k = 0; k < r; ++k) nrm2 += nd[c * r + k];
      const double inv = 1.0 / sqrt(nrm2);
      out = make_float2(static_cast<float>(a * inv), static_cast<float>(b * inv));
    }
  }
  if (act) C[s * r + j] = out;
}

}  // namespace lrq
