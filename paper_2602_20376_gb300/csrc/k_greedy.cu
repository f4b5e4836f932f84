// k_greedy.cu -- greedy local search for Max-K-Cut on a CSR graph, the
// refinement step of the hybrid solver (App. "Hybrid Warm-Start": rank-1
// sweep first, then greedy hill-climbing from its partition).
//
// A vertex i with label z_i and neighbour counts n_i(c) = #{j in N(i), j != i :
// z_j = c} gains g_i = n_i(z_i) - min_{c != z_i} n_i(c) by moving to the label
// of that minimum (ties to the smallest label).  Steepest ascent moves the
// vertex of largest gain.  On the GPU a round moves, at once, every gaining
// vertex that no gaining neighbour outranks, under the strict order (larger
// gain, then smaller index): the moved set is independent, so the gains add
// exactly, and it always contains the steepest move, so every round raises
// the cut and the search ends at a state no single move improves.
//
// A round is two kernels (gains, then moves).  The first round takes every
// vertex; a vertex's gain changes only when it or a neighbour moves, so the
// moves mark those and later rounds recompute the marked ones only.  A thread
// takes a vertex of up to kGrRowMax entries, four gathers in flight; the warp
// takes longer rows together.  Bound: the gathers (first round) and the pass
// over the n marks and gains (later rounds).  n = 10^6, 6.65 * 10^6 entries,
// 16 rounds: gains 264 us (33 the first round), moves 174; 972 and 293 with
// 8 lanes a row and every vertex in every round.
// A graph of up to kGrSmall vertices leaves SMs without rows either way, and a
// round is one chain of dependent reads: there 8 lanes share a row and every
// vertex is taken in every round, without marks.  Whole call, that form / a
// thread a row with marks: n = 1000 258 / 301 us, 5000 290 / 295, 20000 302 /
// 327, 32768 315 / 331; at 50000 the first takes 346, the second 327.
// Rounds are issued in batches of kGrBatch; each round's move count
// lands in a device ring, the next round returns at once when it is zero, and
// the host reads the ring once per batch.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "lrq_device.cuh"
#include "lrq_internal.h"

namespace lrq {

constexpr int kGrThreads = 256;
constexpr int kGrBatch = 8;
constexpr int kGrMaxK = 8;

__device__ __forceinline__ bool gr_row(const int32_t* __restrict__ rowptr, int64_t i, int64_t nnz, int64_t* e0,
                                       int64_t* e1) {
  const int64_t a = rowptr[i], b = rowptr[i + 1];
  *e0 = a;
  *e1 = b;
  return a >= 0 && a <= b && b <= nnz;
}

constexpr int kGrRowMax = 64;  // at most 255: label counts of a thread are bytes
constexpr int64_t kGrSmall = 40960;

__device__ __forceinline__ void gr_store(int64_t i, int zi, int K, const int* cnt, int32_t* __restrict__ gain,
                                         uint8_t* __restrict__ best) {
  int same = 0, bc = -1, bv = 0;
#pragma unroll
  for (int c = 0; c < kGrMaxK; ++c) {
    if (c >= K) break;
    if (c == zi) {
      same = cnt[c];
    } else if (bc < 0 || cnt[c] < bv) {
      bc = c;
      bv = cnt[c];
    }
  }
  const int g = bc >= 0 ? same - bv : 0;
  gain[i] = g > 0 ? g : 0;
  best[i] = static_cast<uint8_t>(g > 0 ? bc : zi);
}

// gain and target label (0 gain when no move helps) of every marked vertex;
// prev NULL: the first round, every vertex.  LR lanes a row; LR > 1 takes every
// vertex and leaves the marks alone.
template <int LR>
__global__ void __launch_bounds__(kGrThreads) gr_gain_kernel(const int32_t* __restrict__ rowptr,
                                                             const int32_t* __restrict__ colidx, int64_t n,
                                                             int64_t nnz, int K, const uint8_t* __restrict__ z,
                                                             int32_t* __restrict__ gain, uint8_t* __restrict__ best,
                                                             uint8_t* __restrict__ dirty,
                                                             const unsigned long long* prev, int32_t* status) {
  if (prev && *prev == 0ull) return;
  constexpr int RW = 32 / LR;  // rows a warp
  const int lane = threadIdx.x & 31, sub = lane % LR;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (kGrThreads / LR);
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * (kGrThreads / LR) + (threadIdx.x >> 5) * RW; i0 < n;
       i0 += stride) {
    const int64_t i = i0 + lane / LR;  // warp-uniform trips
    const bool todo = i < n && (LR > 1 || !prev || dirty[i]);
    if (LR == 1 && i < n && (todo || !prev)) dirty[i] = 0;
    int zi = 0;
    int64_t e0 = 0, e1 = 0;
    bool ok = todo;
    if (todo) {
      zi = z[i];
      if (!gr_row(rowptr, i, nnz, &e0, &e1) || zi >= K) {
        dev_fail(status, LRQ_EINVAL);
        ok = false;
        gain[i] = 0;
        best[i] = static_cast<uint8_t>(zi);
      }
    }
    const bool big = ok && e1 - e0 > kGrRowMax;
    unsigned long long packed = 0;  // eight counts of a byte each
    if (ok && !big) {
      constexpr int U = LR == 1 ? 4 : 1;  // gathers in flight
      for (int64_t e = e0 + sub; e < e1; e += U * LR) {
        int32_t j[U];
        int zj[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          j[u] = e + u < e1 ? colidx[e + u] : static_cast<int32_t>(i);
          if (j[u] < 0 || j[u] >= n) {
            dev_fail(status, LRQ_EINVAL);
            j[u] = static_cast<int32_t>(i);
          }
          zj[u] = j[u] != i ? z[j[u]] : kGrMaxK;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (zj[u] < kGrMaxK) packed += 1ull << (8 * zj[u]);
      }
    }
#pragma unroll
    for (int q = LR / 2; q > 0; q >>= 1) packed += __shfl_xor_sync(0xffffffffu, packed, q);
    if (ok && !big && sub == 0) {
      int cnt[kGrMaxK];
#pragma unroll
      for (int c = 0; c < kGrMaxK; ++c) cnt[c] = static_cast<int>((packed >> (8 * c)) & 0xff);
      gr_store(i, zi, K, cnt, gain, best);
    }
    for (unsigned m = __ballot_sync(0xffffffffu, big && sub == 0); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const int64_t ib = i0 + src / LR, b0 = __shfl_sync(0xffffffffu, e0, src), b1 = __shfl_sync(0xffffffffu, e1, src);
      int cnt[kGrMaxK];
#pragma unroll
      for (int c = 0; c < kGrMaxK; ++c) cnt[c] = 0;
      for (int64_t e = b0 + lane; e < b1; e += 32) {
        const int32_t j = colidx[e];
        if (j < 0 || j >= n) {
          dev_fail(status, LRQ_EINVAL);
          continue;
        }
        if (j == ib) continue;
        const int zj = z[j];
#pragma unroll
        for (int c = 0; c < kGrMaxK; ++c) cnt[c] += (zj == c) ? 1 : 0;
      }
#pragma unroll
      for (int c = 0; c < kGrMaxK; ++c) {
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) cnt[c] += __shfl_xor_sync(0xffffffffu, cnt[c], q);
      }
      if (lane == src) gr_store(ib, zi, K, cnt, gain, best);
    }
  }
}

// move every gaining vertex that no gaining neighbour outranks, and (LR = 1)
// mark it and its neighbours
template <int LR>
__global__ void __launch_bounds__(kGrThreads) gr_move_kernel(const int32_t* __restrict__ rowptr,
                                                             const int32_t* __restrict__ colidx, int64_t n,
                                                             int64_t nnz, const int32_t* __restrict__ gain,
                                                             const uint8_t* __restrict__ best, uint8_t* __restrict__ z,
                                                             uint8_t* __restrict__ dirty,
                                                             const unsigned long long* prev,
                                                             unsigned long long* moved) {
  if (prev && *prev == 0ull) return;
  constexpr int RW = 32 / LR;
  const int lane = threadIdx.x & 31, sub = lane % LR;
  const unsigned row_lanes = ((1u << LR) - 1u) << (lane - sub);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (kGrThreads / LR);
  unsigned mine = 0;
  for (int64_t i0 = static_cast<int64_t>(blockIdx.x) * (kGrThreads / LR) + (threadIdx.x >> 5) * RW; i0 < n;
       i0 += stride) {
    const int64_t i = i0 + lane / LR;
    const int gi = i < n ? gain[i] : 0;
    int64_t e0 = 0, e1 = 0;
    const bool act = gi > 0 && gr_row(rowptr, i, nnz, &e0, &e1);
    const bool big = act && e1 - e0 > kGrRowMax;
    bool blocked = !act || big;
    if (!blocked) {
      constexpr int U = LR == 1 ? 4 : 1;
      for (int64_t e = e0 + sub; e < e1 && !blocked; e += U * LR) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int32_t j = e + u < e1 ? colidx[e + u] : -1;
          if (j < 0 || j >= n || j == i) continue;
          const int gj = gain[j];
          blocked |= gj > gi || (gj == gi && j < i);
        }
      }
    }
    if (LR > 1) blocked = (__ballot_sync(0xffffffffu, blocked) & row_lanes) != 0u;  // a row's lanes agree
    if (!blocked) {
      if (sub == 0) {
        z[i] = best[i];
        ++mine;
      }
      if (LR == 1) {
        dirty[i] = 1;
        for (int64_t e = e0; e < e1; ++e) {
          const int32_t j = colidx[e];
          if (j >= 0 && j < n) dirty[j] = 1;
        }
      }
    }
    for (unsigned m = __ballot_sync(0xffffffffu, big && sub == 0); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const int64_t ib = i0 + src / LR, b0 = __shfl_sync(0xffffffffu, e0, src), b1 = __shfl_sync(0xffffffffu, e1, src);
      const int gb = __shfl_sync(0xffffffffu, gi, src);
      bool out = false;
      for (int64_t e = b0 + lane; e < b1 && !out; e += 32) {
        const int32_t j = colidx[e];
        if (j < 0 || j >= n || j == ib) continue;
        const int gj = gain[j];
        out = gj > gb || (gj == gb && j < ib);
      }
      if (__any_sync(0xffffffffu, out)) continue;
      if (lane == src) {
        z[ib] = best[ib];
        if (LR == 1) dirty[ib] = 1;
        ++mine;
      }
      if (LR == 1) {
        for (int64_t e = b0 + lane; e < b1; e += 32) {
          const int32_t j = colidx[e];
          if (j >= 0 && j < n) dirty[j] = 1;
        }
      }
    }
  }
  mine = __reduce_add_sync(0xffffffffu, mine);
  if (lane == 0 && mine) atomicAdd(moved, static_cast<unsigned long long>(mine));
}

size_t greedy_workspace_bytes(int64_t n) {
  return align_up(sizeof(int32_t) * static_cast<size_t>(n), 256) + 2 * align_up(static_cast<size_t>(n), 256) +
         align_up(sizeof(unsigned long long) * 2 * kGrBatch, 256);
}

int launch_greedy(const int32_t* rowptr, const int32_t* colidx, int64_t n, int64_t nnz, int K, uint8_t* z,
                  int64_t max_rounds, int64_t* cut_out, int64_t* rounds_out, int64_t* moves_out,
                  int32_t* converged_out, void* ws, int32_t* status, cudaStream_t st) {
  char* base = static_cast<char*>(ws);
  int32_t* gain = reinterpret_cast<int32_t*>(base);
  base += align_up(sizeof(int32_t) * static_cast<size_t>(n), 256);
  uint8_t* best = reinterpret_cast<uint8_t*>(base);
  base += align_up(static_cast<size_t>(n), 256);
  uint8_t* dirty = reinterpret_cast<uint8_t*>(base);  // written by the first round
  base += align_up(static_cast<size_t>(n), 256);
  unsigned long long* ring = reinterpret_cast<unsigned long long*>(base);

  const int lanes = n <= kGrSmall ? 8 : 1;
  const auto gr_gain = lanes == 8 ? gr_gain_kernel<8> : gr_gain_kernel<1>;
  const auto gr_move = lanes == 8 ? gr_move_kernel<8> : gr_move_kernel<1>;
  const int blocks =
      static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ceil_div(n * lanes, kGrThreads), 152 * 8)));
  int64_t launched = 0, rounds = 0, moves = 0;
  bool converged = false;
  int e = LRQ_OK;
  for (int64_t b = 0; launched < max_rounds && !converged; ++b) {
    unsigned long long* slot = ring + (b & 1) * kGrBatch;
    if ((e = cuda_check(cudaMemsetAsync(slot, 0, sizeof(unsigned long long) * kGrBatch, st), "memset ring")))
      return e;
    const int nr = static_cast<int>(std::min<int64_t>(kGrBatch, max_rounds - launched));
    for (int t = 0; t < nr; ++t) {
      const unsigned long long* prev =
          (b == 0 && t == 0) ? nullptr : (t == 0 ? ring + ((b - 1) & 1) * kGrBatch + (kGrBatch - 1) : slot + t - 1);
      gr_gain<<<blocks, kGrThreads, 0, st>>>(rowptr, colidx, n, nnz, K, z, gain, best, dirty, prev, status);
      gr_move<<<blocks, kGrThreads, 0, st>>>(rowptr, colidx, n, nnz, gain, best, z, dirty, prev, slot + t);
      count_launch(2);
    }
    if ((e = cuda_check(cudaGetLastError(), "greedy kernels"))) return e;
    unsigned long long hm[kGrBatch];
    int32_t hs = 0;
    if ((e = cuda_check(cudaMemcpyAsync(hm, slot, sizeof(hm), cudaMemcpyDeviceToHost, st), "copy moves"))) return e;
    if ((e = cuda_check(cudaMemcpyAsync(&hs, status, sizeof(int32_t), cudaMemcpyDeviceToHost, st), "copy status")))
      return e;
    if ((e = cuda_check(cudaStreamSynchronize(st), "greedy sync"))) return e;
    if (hs != 0) return fail(hs, "lrq_greedy_cut: the device reported an invalid graph or label");
    for (int t = 0; t < nr; ++t) {
      if (hm[t] == 0) {
        converged = true;
        break;
      }
      ++rounds;
      moves += static_cast<int64_t>(hm[t]);
    }
    launched += nr;
  }
  if (max_rounds == 0) {  // no round ran: validate labels and graph before the cut reads them
    gr_gain<<<blocks, kGrThreads, 0, st>>>(rowptr, colidx, n, nnz, K, z, gain, best, dirty, nullptr, status);
    count_launch();
    int32_t hs = 0;
    if ((e = cuda_check(cudaGetLastError(), "greedy gain kernel"))) return e;
    if ((e = cuda_check(cudaMemcpyAsync(&hs, status, sizeof(int32_t), cudaMemcpyDeviceToHost, st), "copy status")))
      return e;
    if ((e = cuda_check(cudaStreamSynchronize(st), "greedy sync"))) return e;
    if (hs != 0) return fail(hs, "lrq_greedy_cut: the device reported an invalid graph or label");
  }
  if (rounds_out) *rounds_out = rounds;
  if (moves_out) *moves_out = moves;
  if (converged_out) *converged_out = converged ? 1 : 0;
  if (cut_out) return launch_cut_count(rowptr, colidx, n, z, cut_out, st);
  return LRQ_OK;
}

}  // namespace lrq
