// k_graph.cu -- exact Max-K-Cut count on a CSR graph (Sec. 1: K = 3 with a
// Laplacian objective is Max-3-Cut).  cut(z) = #{ {i,j} in E : k_i != k_j },
// each undirected edge counted once, from its lower endpoint, in int64.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

// A thread takes a row of up to kCutRowMax entries with four label gathers in
// flight (they bound it), the warp longer rows together.  Up to kCutSmall
// vertices 8 lanes share a row: a warp then has four long rows to go through
// instead of 32 (2000 rows of 400 entries: 27 us, 79 with a thread a row, 53 without sharing).
constexpr int kCutRowMax = 64;
constexpr int64_t kCutSmall = 40960;

template <int LR>
__global__ void __launch_bounds__(256) cut_count_kernel(const int32_t* __restrict__ rowptr,
                                                        const int32_t* __restrict__ colidx, int64_t n,
                                                        const uint8_t* __restrict__ z,
                                                        unsigned long long* __restrict__ out) {
  constexpr int RW = 32 / LR, U = LR == 1 ? 4 : 1;  // rows a warp, gathers in flight
  __shared__ unsigned long long red[8];
  const int lane = threadIdx.x & 31, sub = lane % LR;
  unsigned long long cnt = 0;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (256 / LR);
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * (256 / LR) + (threadIdx.x >> 5) * RW; i0 < n; i0 += stride) {
    const int64_t i = i0 + lane / LR;  // warp-uniform trips
    uint8_t zi = 0;
    int32_t e0 = 0, e1 = 0;
    if (i < n) {
      zi = z[i];
      e0 = rowptr[i];
      e1 = rowptr[i + 1];
    }
    const bool big = e1 > e0 && static_cast<int64_t>(e1) - e0 > kCutRowMax;
    if (!big) {
      for (int64_t e = static_cast<int64_t>(e0) + sub; e < e1; e += U * LR) {
        int32_t j[U];
        uint8_t zj[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          j[u] = e1 - e > u ? colidx[e + u] : -1;
          zj[u] = j[u] > i ? z[j[u]] : zi;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) cnt += zj[u] != zi ? 1ull : 0ull;
      }
    }
    for (unsigned m = __ballot_sync(0xffffffffu, big && sub == 0); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const int64_t ib = i0 + src / LR, b1 = __shfl_sync(0xffffffffu, e1, src);
      const uint8_t zb = static_cast<uint8_t>(__shfl_sync(0xffffffffu, static_cast<int>(zi), src));
      for (int64_t e = static_cast<int64_t>(__shfl_sync(0xffffffffu, e0, src)) + lane; e < b1; e += 32) {
        const int32_t j = colidx[e];
        cnt += (j > ib && z[j] != zb) ? 1ull : 0ull;
      }
    }
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, m);
  if (lane == 0) red[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) cnt += red[k];
    atomicAdd(out, cnt);
  }
}

int launch_cut_count(const int32_t* rowptr, const int32_t* colidx, int64_t n, const uint8_t* z, int64_t* cut_out,
                     cudaStream_t st) {
  int e = cuda_check(cudaMemsetAsync(cut_out, 0, sizeof(int64_t), st), "cudaMemsetAsync(cut_out)");
  if (e) return e;
  if (n <= 0) return LRQ_OK;
  const int lanes = n <= kCutSmall ? 8 : 1;
  const auto kern = lanes == 8 ? cut_count_kernel<8> : cut_count_kernel<1>;
  const int blocks = static_cast<int>(std::min<int64_t>(ceil_div(n * lanes, 256), 8 * 152));
  kern<<<blocks, 256, 0, st>>>(rowptr, colidx, n, z, reinterpret_cast<unsigned long long*>(cut_out));
  count_launch();
  return cuda_check(cudaGetLastError(), "cut_count_kernel");
}

}  // namespace lrq
