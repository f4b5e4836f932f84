// score_f32x2.cuh -- the FP32 scoring step of one coordinate with packed
// FP32 instructions, shared by the CUDA-core scoring kernel and the batched
// kernel.
//
// sm_103a's fma.rn.f32x2 does two FP32 FMAs a lane in one instruction, each
// rounded like fmaf.  Real and imaginary part are the two halves, so that the
// projection w = V_i c and the update V^H z += conj(V_i) omega^k keep the
// operations and the order of the scalar form (same bits) in half the
// instructions; a row's V is staged as {re, re, im, im} per entry and read
// back as one 16-byte broadcast.  The boundary signs form the byte offset of
// omega^k in a table with one entry per sign pattern, so no code is computed.
// What binds next are the shared-memory reads: an SM returns 128 bytes a cycle,
// 4 cycles for a 16-byte read of a warp whatever it broadcasts, so a row's
// entries are read once for several candidates of a thread and the table entry
// is 8 bytes.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lrq_device.cuh"

namespace lrq {

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }

// hi += v m for a pair of multipliers in {-1, 0, 1}; returns the rounding error
// (exact two-sum)
__device__ __forceinline__ f32x2 add_unit(f32x2& hi, f32x2 v, f32x2 m) {
  const f32x2 s = fma2(v, m, hi);
  const f32x2 nb = add2(hi, neg2(s));  // minus the part of v m that reached s
  const f32x2 t = add2(s, nb);
  const f32x2 e = add2(add2(hi, neg2(t)), fma2(v, m, nb));
  hi = s;
  return e;
}

// Decision boundaries theta_m = pi(2m+1)/K in FP32, the first (B_K + 1) / 2 of
// them: the others are mirror images (odd K: m and K-1-m share cos and have
// opposite sin; even K: m and K/2-1-m share sin and have opposite cos).  The
// same values as make_alphabet's FP32 tables.
template <int K>
__host__ __device__ constexpr float boundary_cos(int m) {
  if (K == 2) {
    constexpr float t[] = {0.f};
    return t[m];
  }
  if (K == 3) {
    constexpr float t[] = {0x1p-1f, -1.f};
    return t[m];
  }
  if (K == 4) {
    constexpr float t[] = {0x1.6a09e6p-1f};
    return t[m];
  }
  if (K == 5) {
    constexpr float t[] = {0x1.9e377ap-1f, -0x1.3c6ef4p-2f, -1.f};
    return t[m];
  }
  if (K == 6) {
    constexpr float t[] = {0x1.bb67aep-1f, 0.f};
    return t[m];
  }
  if (K == 7) {
    constexpr float t[] = {0x1.cd4bcap-1f, 0x1.c7b90ep-3f, -0x1.3f3a0ep-1f, -1.f};
    return t[m];
  }
  if (K == 8) {
    constexpr float t[] = {0x1.d906bcp-1f, 0x1.87de2ap-2f};
    return t[m];
  }
  return 0.f;
}
template <int K>
__host__ __device__ constexpr float boundary_sin(int m) {
  if (K == 2) {
    constexpr float t[] = {1.f};
    return t[m];
  }
  if (K == 3) {
    constexpr float t[] = {0x1.bb67aep-1f, 0.f};
    return t[m];
  }
  if (K == 4) {
    constexpr float t[] = {0x1.6a09e6p-1f};
    return t[m];
  }
  if (K == 5) {
    constexpr float t[] = {0x1.2cf23p-1f, 0x1.e6f0e2p-1f, 0.f};
    return t[m];
  }
  if (K == 6) {
    constexpr float t[] = {0x1p-1f, 1.f};
    return t[m];
  }
  if (K == 7) {
    constexpr float t[] = {0x1.bc4c04p-2f, 0x1.f329cp-1f, 0x1.904c38p-1f, 0.f};
    return t[m];
  }
  if (K == 8) {
    constexpr float t[] = {0x1.87de2ap-2f, 0x1.d906bcp-1f};
    return t[m];
  }
  return 0.f;
}

// Sign pattern of the boundary projections p_m = y cos - x sin > 0 (the same
// roundings as decide_fp32), times 8: a byte offset into the z table.
template <int K>
__device__ __forceinline__ uint32_t sign_offset(float x, float y) {
  constexpr int BK = (K % 2 == 0) ? K / 2 : K;
  uint32_t off = 0;
#pragma unroll
  for (int m = 0; m < (BK + 1) / 2; ++m) {
    const float c = boundary_cos<K>(m), s = boundary_sin<K>(m);
    const int mm = BK - 1 - m;
    float p, q;
    if (s == 0.f) {  // the boundary on the negative real axis
      p = q = -y;
    } else if (c == 0.f) {  // the boundary on the imaginary axis
      p = q = -x;
    } else {
      const float t = x * s;
      p = fmaf(y, c, -t);
      q = K % 2 == 1 ? fmaf(y, c, t) : fmaf(y, -c, -t);
    }
    if (p > 0.f) off |= 8u << m;
    if (mm != m && q > 0.f) off |= 8u << mm;
  }
  return off;
}

// Sign pattern [p_m > 0] (bit m) and the smallest |p_m|, with the roundings of
// decide_fp32.
template <int K>
__device__ __forceinline__ uint32_t sign_lines(float x, float y, float* pmin) {
  constexpr int BK = (K % 2 == 0) ? K / 2 : K;
  uint32_t bits = 0;
  float mn = INFINITY;
#pragma unroll
  for (int m = 0; m < (BK + 1) / 2; ++m) {
    const float c = boundary_cos<K>(m), s = boundary_sin<K>(m);
    const int mm = BK - 1 - m;
    float p, q;
    if (s == 0.f) {
      p = q = -y;
    } else if (c == 0.f) {
      p = q = -x;
    } else {
      const float t = x * s;
      p = fmaf(y, c, -t);
      q = K % 2 == 1 ? fmaf(y, c, t) : fmaf(y, -c, -t);
    }
    if (p > 0.f) bits |= 1u << m;
    mn = fminf(mn, fabsf(p));
    if (mm != m) {
      if (q > 0.f) bits |= 1u << mm;
      mn = fminf(mn, fabsf(q));
    }
  }
  *pmin = mn;
  return bits;
}

// Certificate of an FP32 decision.  The error of a boundary projection is below
// gamma sum_j |V_ij|_1 |c_j|_1 (|x|_1 = |Re| + |Im|), gamma = (2 r + 4) 2 u + 8 u
// with u = 2^-24, plus a few roundings of 2^-150 where products underflow;
// |c_j|_1 is replaced by its largest value, so that the bound of an evaluation is
// one FMA: fp32_proj_bound(fp32_row_bound(sum_j |V_ij|_1), fp32_dir_bound(max
// |c_j|_1, r)).  Rows and directions whose products could overflow (sums or
// components above 2^62), and directions too small for the product to hold the
// bound, get an infinite one.
__device__ __forceinline__ float fp32_row_bound(float ab) { return ab < 0x1p62f ? ab : INFINITY; }
__device__ __forceinline__ float fp32_dir_bound(float mx, int r) {
  return mx < 0x1p62f && mx > 0x1p-100f ? mx * (static_cast<float>(2 * r + 4) * 2.0f + 12.0f) * 5.9604644775390625e-08f : INFINITY;
}
__device__ __forceinline__ float fp32_proj_bound(float row, float dir) { return fmaf(row, dir, 0x1p-140f); }

// A sign pattern whose code is k.
template <int K>
__device__ __forceinline__ uint32_t pattern_of(int k) {
  if constexpr (K % 2 == 0) {
    // w in sector k lies beyond boundaries 0..k-1 (mod K/2, the other side past half a turn)
    constexpr int H = K / 2;
    return k <= H ? (1u << k) - 1u : ((1u << H) - 1u) ^ ((1u << (k - H)) - 1u);
  } else {
    return k == 0 ? 0u : 1u << (k - 1);
  }
}

// K as a template argument: 2..8, kAnyK8 for an alphabet of at most 8 known at
// run time, 0 for larger ones.
constexpr int kAnyK8 = -1;

// entries of the z table (sign patterns; codes where K is known at run time only)
// and its filling by a block's threads
template <int K>
struct ZTable {
  static constexpr int kEntries = K <= 0 ? kMaxK : 1 << ((K % 2 == 0) ? K / 2 : K);
};
template <int K>
__device__ __forceinline__ void fill_ztable(float2* zt, const float* zr, const float* zi, int Kdyn) {
  const int count = K <= 0 ? Kdyn : ZTable<K>::kEntries;
  for (int t = threadIdx.x; t < count; t += blockDim.x) {
    int k = t;
    if constexpr (K > 0) k = decide_from_signs<K>(static_cast<uint32_t>(t));
    zt[t] = make_float2(zr[k], zi[k]);
  }
}

// One candidate's direction: {cr, ci} and {-ci, cr} per component.
template <int R>
struct Dir2 {
  f32x2 a[R], b[R];
  __device__ __forceinline__ void set(int j, float2 c) {
    a[j] = pack2(c.x, c.y);
    b[j] = pack2(-c.y, c.x);
  }
};

// The sign rule of decide_fp32 for K <= 8 known at run time.  bc, bs: the first
// (B_K + 1) / 2 boundaries (the others are their mirror images, as above), in
// registers: read from memory line by line they took the batched kernel twice
// its time at K = 5.
constexpr int kAnyLines = 4;
__device__ __forceinline__ int decide_any8(float x, float y, int K, const float (&bc)[kAnyLines],
                                           const float (&bs)[kAnyLines]) {
  const bool odd = K % 2 == 1;
  const int BK = odd ? K : K / 2;
  uint32_t sb = 0;
#pragma unroll
  for (int m = 0; m < kAnyLines; ++m) {
    if (2 * m < BK) {
      const float t = x * bs[m], q = fmaf(y, bc[m], t);
      if (fmaf(y, bc[m], -t) > 0.f) sb |= 1u << m;
      if ((odd ? q : -q) > 0.f) sb |= 1u << (BK - 1 - m);
    }
  }
  if (!odd) {
    const int c = __popc(sb);
    return (sb & 1u) ? c : (c == 0 ? 0 : K - c);
  }
  const uint32_t t = sb & ~(sb >> 1) & ((1u << (K - 1)) - 1u);
  return t ? __ffs(t) : 0;
}

// acc[j] += conj(V_ij) z_i for one candidate; v: the row's {re, re, im, im}.
// bc, bs: kAnyK8's boundaries.  VFIRST: the order of the two products of w (each caller's own).
template <int K, int R, bool VFIRST>
__device__ __forceinline__ void score_row(const ulonglong2 (&v)[R], const Dir2<R>& d, const float2* zt, int Kdyn,
                                          const float (&bc)[kAnyLines], const float (&bs)[kAnyLines],
                                          f32x2 (&acc)[R]) {
  f32x2 w = 0;  // {0, 0}
#pragma unroll
  for (int j = 0; j < R; ++j) {
    if constexpr (VFIRST) {
      w = fma2(v[j].x, d.a[j], w);
      w = fma2(v[j].y, d.b[j], w);
    } else {
      w = fma2(v[j].y, d.b[j], w);
      w = fma2(v[j].x, d.a[j], w);
    }
  }
  float x, y;
  unpack2(w, x, y);
  uint32_t off;
  if constexpr (K > 0)
    off = sign_offset<K>(x, y);
  else
    off = 8u * static_cast<uint32_t>(K == 0 ? decide_fp32_generic(x, y, Kdyn) : decide_any8(x, y, Kdyn, bc, bs));
  const float2 z = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(zt) + off);
  const f32x2 za = pack2(z.x, z.y), zb = pack2(z.y, -z.x);
#pragma unroll
  for (int j = 0; j < R; ++j) {
    acc[j] = fma2(v[j].y, zb, acc[j]);
    acc[j] = fma2(v[j].x, za, acc[j]);
  }
}

// The same in scalar FMAs on the row's {re, im} (same operations and order), for K >
// 8: the angle is most of an evaluation there and half the shared-memory reads count
// for more than half the FMAs.
template <int R, bool VFIRST>
__device__ __forceinline__ void score_row_scalar(const float2 (&v)[R], const float2 (&c)[R], const float2* zt, int K,
                                                 float2 (&acc)[R]) {
  float x = 0.f, y = 0.f;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    if constexpr (VFIRST) {
      x = fmaf(-v[j].y, c[j].y, fmaf(v[j].x, c[j].x, x));
      y = fmaf(v[j].y, c[j].x, fmaf(v[j].x, c[j].y, y));
    } else {
      x = fmaf(v[j].x, c[j].x, fmaf(-v[j].y, c[j].y, x));
      y = fmaf(v[j].x, c[j].y, fmaf(v[j].y, c[j].x, y));
    }
  }
  const float2 z = zt[decide_fp32_generic(x, y, K)];
#pragma unroll
  for (int j = 0; j < R; ++j) {
    acc[j].x = fmaf(v[j].x, z.x, fmaf(v[j].y, z.y, acc[j].x));
    acc[j].y = fmaf(v[j].x, z.y, fmaf(-v[j].y, z.x, acc[j].y));
  }
}

}  // namespace lrq
