// k_select.cu -- top-m selection of scored candidates ("returns only the best
// candidate found", Sec. 5; best-of-S, Sec. 4.2), generalised to the m best
// for the FP64 re-scoring step.
//
// Keys are 64-bit: the FP32 score bits (scores are >= 0, so their bit
// patterns order like the values) above 0xFFFFFFFF - index, so the key order
// is "larger score first, then smaller index".  Each pass sorts segments of
// kSeg keys with a bitonic network (descending) and keeps the first m of every
// segment; passes repeat until one segment remains.  A thread holds two
// neighbouring keys: of the network's 66 steps 51 exchange within a warp by
// shuffles and 15 through shared memory (all in shared memory, a barrier each:
// 17.9 us a segment, now 7.0).
#include <cuda_runtime.h>
#include <stdint.h>

#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

constexpr int kSeg = 2048;
constexpr int kSelThreads = 1024;

static_assert(kSeg == 2 * kSelThreads, "two keys per thread");

// the larger of the pair where `up`, else the smaller
__device__ __forceinline__ uint64_t sel_keep(uint64_t a, uint64_t b, bool up) { return (a > b) == up ? a : b; }

__global__ void __launch_bounds__(kSelThreads) topm_pass_kernel(const uint64_t* __restrict__ in, int64_t count,
                                                                int m, uint64_t* __restrict__ out,
                                                                int64_t* __restrict__ top_idx,
                                                                float* __restrict__ top_f) {
  __shared__ __align__(16) ulonglong2 sk[2][kSelThreads];
  const int t = threadIdx.x;
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kSeg + 2 * t;
  uint64_t k0 = base < count ? in[base] : 0ull, k1 = base + 1 < count ? in[base + 1] : 0ull;
  int buf = 0;
  // bitonic sort of positions 2 t, 2 t + 1, descending
#pragma unroll
  for (int size = 2; size <= kSeg; size <<= 1) {
    const bool desc = ((2 * t) & size) == 0;
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride == 1) {
        const uint64_t a = sel_keep(k0, k1, desc);
        k1 = sel_keep(k0, k1, !desc);
        k0 = a;
        continue;
      }
      const int x = stride >> 1;  // the partner thread holds the same half of its pair
      const bool up = ((t & x) == 0) == desc;
      uint64_t o0, o1;
      if (x < 32) {
        o0 = __shfl_xor_sync(0xffffffffu, k0, x);
        o1 = __shfl_xor_sync(0xffffffffu, k1, x);
      } else {  // two buffers: one barrier a step
        sk[buf][t] = make_ulonglong2(k0, k1);
        __syncthreads();
        const ulonglong2 o = sk[buf][t ^ x];
        o0 = o.x;
        o1 = o.y;
        buf ^= 1;
      }
      k0 = sel_keep(k0, o0, up);
      k1 = sel_keep(k1, o1, up);
    }
  }
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int pos = 2 * t + e;
    const uint64_t k = e ? k1 : k0;
    if (pos >= m) continue;
    if (top_idx) {  // final pass: decode
      top_idx[pos] = static_cast<int64_t>(0xFFFFFFFFu - static_cast<uint32_t>(k & 0xFFFFFFFFull));
      top_f[pos] = __uint_as_float(static_cast<uint32_t>(k >> 32));
    } else {
      out[static_cast<int64_t>(blockIdx.x) * m + pos] = k;
    }
  }
}

size_t topm_scratch_keys(int64_t count, int m) {
  // two ping-pong buffers, each large enough for the first pass output
  int64_t segs = ceil_div(count, kSeg);
  return static_cast<size_t>(2 * segs * m);
}

int launch_topm(const uint64_t* keys_in, int64_t count, int m, uint64_t* scratch, int64_t* top_idx, float* top_f,
                cudaStream_t st) {
  if (m < 1 || m > kSeg / 4) return fail(LRQ_EUNSUPPORTED, "top_m out of range");
  int64_t segs0 = ceil_div(count, kSeg);
  uint64_t* buf[2] = {scratch, scratch + segs0 * m};
  const uint64_t* src = keys_in;
  int64_t cnt = count;
  int which = 0;
  for (;;) {
    int64_t segs = ceil_div(cnt, kSeg);
    if (segs <= 1) {
      topm_pass_kernel<<<1, kSelThreads, 0, st>>>(src, cnt, m, nullptr, top_idx, top_f);
      count_launch();
      return cuda_check(cudaGetLastError(), "topm_pass_kernel(final)");
    }
    topm_pass_kernel<<<static_cast<unsigned>(segs), kSelThreads, 0, st>>>(src, cnt, m, buf[which], nullptr,
                                                                          nullptr);
    count_launch();
    int e = cuda_check(cudaGetLastError(), "topm_pass_kernel");
    if (e) return e;
    src = buf[which];
    cnt = segs * m;
    which ^= 1;
  }
}

}  // namespace lrq
