// k_mlp_tc.cu -- the learned proposal's GEMMs in BF16 mode on the tensor
// cores (tcgen05): C = act(op(A) op(B) + bias), optionally zeroed where
// mask <= 0, with op(A) M x K and op(B) K x N, either stored transposed.
// The operands are rounded to bfloat16 (nearest even) as they are staged and
// the products accumulate in FP32 in tensor memory.
//
// One CTA of eight warps per 128 x BN output tile, BN = 32 or 64.  The whole of
// K up to 256 is staged at once (all its loads in flight together), then
// multiplied: op(A) (128 rows) and op(B) transposed (BN rows) go into shared
// memory as bfloat16 in the no-swizzle K-major core-matrix order (8 rows x 16
// bytes per core matrix; per MMA of K = 16, the rows' K 0..7 for all rows,
// then K 8..15), a thread converting eight consecutive K of a row into one
// 16-byte store; the stores are made visible to the tensor core, and one
// elected thread issues a tcgen05.mma kind::f16 (BF16 x BF16 -> FP32, M 128,
// N BN) per 16 of K and commits them to an mbarrier that every thread waits
// for.  Rows past M and columns past N are neither loaded nor written: they
// reach no output in range.  Epilogue: warp w reads 32 tensor-memory lanes
// (rows 32 (w % 4)) x half of the columns and adds the bias, applies ReLU and
// the mask.
// Bound: latency (at a batch of 64 a GEMM is under 1 us of loads and 0.1 of
// MMAs); chunks of 64 along K with 64 scalar loads a thread, each chunk
// waiting for its own loads and MMAs, took 21 us a GEMM, now 7.5.  BN = 32
// while BN = 64 would leave SMs without a tile: the three layers forward with BN = 32 /
// 64 take 36 / 41 us at a batch of 64, 39 / 45 at 2048, 47 / 46 at 4096 (128 tiles of
// 64), 60 / 52 at 6000, 143 / 116 at 20000.
// The wait is bounded (~1 s); if it runs out (never observed) the kernel
// records the fault, writes NaN into its tile, waits (bounded) for its MMAs,
// frees its tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lrq_device.cuh"
#include "lrq_internal.h"
#include "ptx_sm100.cuh"

namespace lrq {

constexpr int kMgM = 128, kMgK = 256, kMgThreads = 256;
constexpr long long kMgWait = 2000000000LL;

__device__ int32_t g_mlp_tc_fault = 0;

// Eight consecutive K of one row of an operand as bfloat16 (zero past K).
// along_k: K is the contiguous direction (stride 1), else rows are and K has
// stride ld; vec: the row's K may be read 16 bytes at a time.
__device__ __forceinline__ uint4 mg_load8(const float* __restrict__ p, int row, int gk, int K, int ld, bool along_k,
                                          bool vec) {
  float v[8];
  if (along_k) {
    const float* q = p + static_cast<int64_t>(row) * ld + gk;
    if (vec && gk + 8 <= K) {
      const float4 a = reinterpret_cast<const float4*>(q)[0], b = reinterpret_cast<const float4*>(q)[1];
      v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = gk + e < K ? q[e] : 0.f;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = gk + e < K ? p[static_cast<int64_t>(gk + e) * ld + row] : 0.f;
  }
  __align__(16) __nv_bfloat16 h[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) h[e] = __float2bfloat16_rn(v[e]);
  return *reinterpret_cast<uint4*>(h);
}

template <int BN>
__global__ void __launch_bounds__(kMgThreads) mlp_gemm_tc_kernel(int M, int N, int K, const float* __restrict__ A,
                                                                 int lda, int ta, int va, const float* __restrict__ Bm,
                                                                 int ldb, int tb, int vb,
                                                                 const float* __restrict__ bias, int relu,
                                                                 const float* __restrict__ mask,
                                                                 float* __restrict__ C, int ldc, int vc) {
  extern __shared__ __align__(1024) uint8_t mg_smem[];
  uint4* sa = reinterpret_cast<uint4*>(mg_smem);                 // [K / 8][128 rows]
  uint4* sb = sa + kMgM * kMgK / 8;                              // [K / 8][BN rows]
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int row0 = blockIdx.y * kMgM, col0 = blockIdx.x * BN;
  if (tid == 0) {
    ptx::mbar_init(&bar, 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(&tmem_slot, BN);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const uint32_t sa_u = ptx::smem_u32(sa), sb_u = ptx::smem_u32(sb);
  constexpr uint32_t idesc = ptx::idesc_bf16_f32(kMgM, BN);
  volatile int never = 0;
  bool ok = true;
  uint32_t phase = 0;
  const int rows = min(kMgM, M - row0), cols = min(BN, N - col0);
  for (int k0 = 0; k0 < K && ok; k0 += kMgK) {
    const int k16 = (min(kMgK, K - k0) + 15) / 16;  // MMAs of this chunk
    const int k8 = 2 * k16;
    // lanes take consecutive rows: a row's eight K are one or two sectors, and
    // the stores are contiguous
#pragma unroll 4
    for (int t = tid; t < k8 * kMgM; t += kMgThreads) {
      const int i = t & (kMgM - 1), c = t / kMgM;
      if (i < rows) sa[c * kMgM + i] = mg_load8(A, row0 + i, k0 + 8 * c, K, lda, !ta, va);
    }
#pragma unroll 4
    for (int t = tid; t < k8 * BN; t += kMgThreads) {
      const int j = t & (BN - 1), c = t / BN;
      if (j < cols) sb[c * BN + j] = mg_load8(Bm, col0 + j, k0 + 8 * c, K, ldb, tb, vb);
    }
    ptx::fence_proxy_async_smem();  // the staged operands, visible to the tensor core
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
      ptx::tc_fence_after();
      for (int q = 0; q < k16; ++q) {
        const uint64_t ad = ptx::smem_desc(sa_u + q * 2 * kMgM * 16, kMgM * 16, 128);
        const uint64_t bd = ptx::smem_desc(sb_u + q * 2 * BN * 16, BN * 16, 128);
        ptx::mma_f16_ss_elect(tmem, ad, bd, idesc, (k0 > 0 || q > 0) ? 1u : 0u);
      }
      ptx::mma_commit_elect(&bar);
    }
    // the chunk's MMAs (and their reads of the buffers) are complete
    const bool done = ptx::mbar_wait(&bar, phase, &never, kMgWait);
    ok = __syncthreads_and(done) != 0;
    phase ^= 1u;
    ptx::tc_fence_after();
  }
  const int quad = warp & 3, half = warp >> 2;
  const int gi = row0 + quad * 32 + lane;
  if (ok) {
#pragma unroll
    for (int c0 = half * (BN / 2); c0 < (half + 1) * (BN / 2); c0 += 16) {
      uint32_t v[16];
      ptx::tmem_ld_x16(tmem + (static_cast<uint32_t>(quad * 32) << 16) + c0, v);
      ptx::tmem_wait_ld();
      if (gi < M) {
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
          const int gj = col0 + c0 + c;
          float x[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            x[e] = __uint_as_float(v[c + e]);
            if (gj + e < N) {
              x[e] += bias ? bias[gj + e] : 0.f;
              if (relu) x[e] = fmaxf(x[e], 0.f);
              if (mask && !(mask[static_cast<int64_t>(gi) * ldc + gj + e] > 0.f)) x[e] = 0.f;
            }
          }
          float* out = C + static_cast<int64_t>(gi) * ldc + gj;
          if (vc && gj + 4 <= N) {
            *reinterpret_cast<float4*>(out) = make_float4(x[0], x[1], x[2], x[3]);
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (gj + e < N) out[e] = x[e];
          }
        }
      }
    }
  } else {
    if (tid == 0) atomicExch(&g_mlp_tc_fault, 1);
    if (half == 0 && gi < M)
      for (int gj = col0; gj < col0 + BN && gj < N; ++gj) C[static_cast<int64_t>(gi) * ldc + gj] = __int_as_float(0x7fc00000);
    // the MMAs still in flight complete before the tensor memory and the
    // shared buffers are released
    ptx::mbar_wait(&bar, phase ^ 1u, &never, kMgWait);
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, BN);
  }
}

template <int BN>
static int mg_launch(cudaStream_t st, int M, int N, int K, const float* A, int lda, int ta, const float* Bm, int ldb,
                     int tb, const float* bias, int relu, const float* mask, float* C, int ldc) {
  // 80 or 96 KB of operands: two CTAs per SM at most, so their tensor-memory
  // allocations always fit
  constexpr int smem = (kMgM + BN) * kMgK * 2;
  const int e = cuda_check(cudaFuncSetAttribute(mlp_gemm_tc_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                smem),
                           "cudaFuncSetAttribute(mlp_gemm_tc_kernel)");
  if (e) return e;
  auto aligned = [](const void* p, int ld) { return reinterpret_cast<uintptr_t>(p) % 16 == 0 && ld % 4 == 0 ? 1 : 0; };
  dim3 grid(static_cast<unsigned>(ceil_div(N, BN)), static_cast<unsigned>(ceil_div(M, kMgM)));
  mlp_gemm_tc_kernel<BN><<<grid, kMgThreads, smem, st>>>(M, N, K, A, lda, ta, aligned(A, lda), Bm, ldb, tb,
                                                         aligned(Bm, ldb), bias, relu, mask, C, ldc, aligned(C, ldc));
  count_launch();
  return LRQ_OK;
}

int launch_mlp_gemm_tc(cudaStream_t st, int M, int N, int K, const float* A, int lda, int ta, const float* Bm,
                       int ldb, int tb, const float* bias, int relu, const float* mask, float* C, int ldc) {
  if (ceil_div(M, kMgM) * ceil_div(N, 64) < num_sms_current())
    return mg_launch<32>(st, M, N, K, A, lda, ta, Bm, ldb, tb, bias, relu, mask, C, ldc);
  return mg_launch<64>(st, M, N, K, A, lda, ta, Bm, ldb, tb, bias, relu, mask, C, ldc);
}

}  // namespace lrq
