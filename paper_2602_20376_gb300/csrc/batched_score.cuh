// batched_score.cuh -- the persistent scoring kernel of the batched launch
// (k_batched.cu): its problem descriptors, work items and both forms' template.
// The forms, one and four slots a thread, are compiled in k_batched_wide.cu and
// k_batched_four.cu, side by side.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "enum_device.cuh"
#include "lrq_device.cuh"
#include "lrq_internal.h"
#include "score_f32x2.cuh"

namespace lrq {

constexpr int kBSlots = 256;      // candidate x row group slots of a block
constexpr int kBRows = 128;       // V rows per shared-memory stage
constexpr int kBEnumChunk = 1024;  // index sets per exact work item

struct BProb {
  const float2* V;
  const float2* C;  // directions: the caller's, or the workspace slot when drawn
  int64_t n;
  int r, K, S, tile;
  int gen;          // 1: draw C from seed (+ epoch)
  int exact;        // 1: solved exactly by vertex enumeration (S = 0)
  uint64_t seed;
  int64_t key_off;  // offset of the problem's selection keys
  int64_t eb_off;   // exact: offset of its chunk results
  int nchunks;      // exact: work items
  int pad;
  unsigned long long lvl_total[kEnumMaxD];  // exact: index sets of level d at [d - 1]
};

struct BItem {
  int p;
  int s0;
};

struct BTable {
  float bcos[8], bsin[8];
  float zr[kMaxK], zi[kMaxK];
  double bcos64[8], bsin64[8];
  double zr64[kMaxK], zi64[kMaxK];
};

// ---------------------------------------------------------------------------
// persistent scoring kernel
// ---------------------------------------------------------------------------
constexpr int kBZTable = 128;  // ZTable<7>, the largest

// The slots' FP64 sums: while a thread takes its four slots at once (r <= 4,
// where the first 24 KB hold sums and staged rows) they stay in shared memory
// over the stages; for larger r they take the staged rows' place at the end.
struct BShared {
  union {
    struct {
      double sums[kBSlots * 8];             // r <= 4: [2 r][slot]
      float4 vs[kBRows * 4];                // {re, re, im, im} per entry (score_f32x2.cuh)
    } small;
    float4 vs[kBRows * kMaxRank];
    double comb[kBSlots * 2 * kMaxRank];    // [slot][2 r]
  };
  float2 zt[kBZTable];                      // z table: an entry per sign pattern or code
  int next;
};

// A thread scores candidates s0 + cl + q T / PT, q < PT, on row group g: all on
// every row it reads (r <= 4), or a part of them at a time on the staged rows
// (their directions re-read, their FP64 sums in local memory).
// Bound: FP32 FMAs and shared-memory reads, as score_fp32_kernel; 512 uneven
// instances of up to 8192 directions: 11.0 ms, 15.3 with one candidate per thread
// and scalar FMAs, 11.7 with two.
template <int R, int KC, int PT>
__device__ void b_score_item(const BProb& pb, const BTable& tb, int s0, BShared& sh, uint64_t* __restrict__ keys) {
  constexpr int NT = kBSlots / PT;  // threads
  static_assert(ZTable<KC>::kEntries <= kBZTable, "the z table holds every pattern");
  constexpr int P = R <= 4 || PT == 1 ? PT : (R <= 6 ? 2 : 1);  // candidates at once
  constexpr bool kShared = R <= 4;
  const int T = pb.tile, H = T / PT, RS = kBSlots / T;
  const int tid = threadIdx.x, cl = tid % H, g = tid / H;
  float4* const vs = kShared ? sh.small.vs : sh.vs;
  float bc[kAnyLines], bs[kAnyLines];
#pragma unroll
  for (int m = 0; m < kAnyLines; ++m) {
    bc[m] = KC == kAnyK8 ? tb.bcos[m] : 0.f;
    bs[m] = KC == kAnyK8 ? tb.bsin[m] : 0.f;
  }
  Dir2<R> d[P];
  auto load_dirs = [&](int q0) {
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const int s = s0 + cl + (q0 + q) * H;
#pragma unroll
      for (int j = 0; j < R; ++j)
        d[q].set(j, s < pb.S ? pb.C[static_cast<int64_t>(s) * R + j] : make_float2(0.f, 0.f));
    }
  };
  double acc64[kShared ? 1 : PT][2 * R];
  auto slot = [&](int q) { return g * T + cl + q * H; };
  if constexpr (kShared) {
    load_dirs(0);
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
      for (int j = 0; j < 2 * R; ++j) sh.small.sums[j * kBSlots + slot(q)] = 0.0;
  } else {
    for (int q = 0; q < PT; ++q)
#pragma unroll
      for (int j = 0; j < 2 * R; ++j) acc64[q][j] = 0.0;
  }
  fill_ztable<KC>(sh.zt, tb.zr, tb.zi, pb.K);
  for (int64_t b0 = 0; b0 < pb.n; b0 += kBRows) {
    const int rows = static_cast<int>(min(static_cast<int64_t>(kBRows), pb.n - b0));
    __syncthreads();
#pragma unroll 4
    for (int t = tid; t < rows * R; t += NT) {
      const float2 v = pb.V[b0 * R + t];
      vs[t] = make_float4(v.x, v.x, v.y, v.y);
    }
    __syncthreads();
#pragma unroll 1
    for (int q0 = 0; q0 < PT; q0 += P) {
      if constexpr (!kShared) load_dirs(q0);
      f32x2 acc[P][R];
#pragma unroll
      for (int q = 0; q < P; ++q)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[q][j] = 0;
#pragma unroll 1
      for (int i = g; i < rows; i += RS) {
        ulonglong2 v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = reinterpret_cast<const ulonglong2*>(vs)[i * R + j];
#pragma unroll
        for (int q = 0; q < P; ++q)
          score_row<KC, R, false>(v, d[q], sh.zt, pb.K, bc, bs, acc[q]);
      }
#pragma unroll
      for (int q = 0; q < P; ++q)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          float re, im;
          unpack2(acc[q][j], re, im);
          if constexpr (kShared) {
            sh.small.sums[2 * j * kBSlots + slot(q)] += static_cast<double>(re);
            sh.small.sums[(2 * j + 1) * kBSlots + slot(q)] += static_cast<double>(im);
          } else {
            acc64[q0 + q][2 * j] += static_cast<double>(re);
            acc64[q0 + q][2 * j + 1] += static_cast<double>(im);
          }
        }
    }
  }
  __syncthreads();
  if constexpr (!kShared) {
    for (int q = 0; q < PT; ++q)
#pragma unroll
      for (int j = 0; j < 2 * R; ++j) sh.comb[slot(q) * (2 * R) + j] = acc64[q][j];
    __syncthreads();
  }
  for (int c = tid; c < T; c += NT) {
    const int s = s0 + c;
    if (s >= pb.S) break;
    double f = 0.0;
#pragma unroll
    for (int j = 0; j < 2 * R; ++j) {
      double v = 0.0;
      for (int gg = 0; gg < RS; ++gg)
        v += kShared ? sh.small.sums[j * kBSlots + gg * T + c] : sh.comb[(gg * T + c) * (2 * R) + j];
      f += v * v;
    }
    const uint32_t fb = __float_as_uint(static_cast<float>(f));
    keys[pb.key_off + s] = (static_cast<uint64_t>(fb) << 32) | static_cast<uint64_t>(0xFFFFFFFFu - static_cast<uint32_t>(s));
  }
}

// K = 5, 6, 7 have code of their own only in the form that batches of mostly
// these take (b_slots_per_thread): every alphabet costs both files compile time.
template <int R, int PT>
__device__ __forceinline__ void b_dispatch_k(const BProb& pb, const BTable& tb, int s0, BShared& sh,
                                             uint64_t* keys) {
  switch (pb.K) {
    case 2: b_score_item<R, 2, PT>(pb, tb, s0, sh, keys); break;
    case 3: b_score_item<R, 3, PT>(pb, tb, s0, sh, keys); break;
    case 4: b_score_item<R, 4, PT>(pb, tb, s0, sh, keys); break;
    case 8: b_score_item<R, 8, PT>(pb, tb, s0, sh, keys); break;
    case 5: b_score_item<R, PT == 1 ? 5 : kAnyK8, PT>(pb, tb, s0, sh, keys); break;
    case 6: b_score_item<R, PT == 1 ? 6 : kAnyK8, PT>(pb, tb, s0, sh, keys); break;
    case 7: b_score_item<R, PT == 1 ? 7 : kAnyK8, PT>(pb, tb, s0, sh, keys); break;
    default: b_score_item<R, 0, PT>(pb, tb, s0, sh, keys); break;
  }
}

// One exact work item: index sets [chunk kBEnumChunk, (chunk + 1) kBEnumChunk)
// of the problem's levels d = r..1 taken in turn, kBEnumChunk / NT
// consecutive ranks per thread; the block's best candidate (the solver's
// order) goes to ebest[eb_off + chunk].  Kept out of line so that the
// scoring path keeps its registers.
template <int NT>
__device__ __noinline__ void b_enum_item(const BProb& pb, const EnumTables& tb, int chunk, BShared& sh,
                                         EnumBest* __restrict__ ebest, int32_t* status) {
  constexpr int kRanks = kBEnumChunk / NT;
  const EnumV32 va{pb.V, pb.r};
  const int n = static_cast<int>(pb.n);
  const int N = n * tb.BK;
  unsigned long long total = 0;
  for (int d = 1; d <= pb.r; ++d) total += pb.lvl_total[d - 1];
  EnumBest best;
  best.f = -1.0;
  best.level = 0;
  best.sign = 1;
  best.rank = 0;
  best.choice = 0;
  unsigned long long q = static_cast<unsigned long long>(chunk) * kBEnumChunk +
                         static_cast<unsigned long long>(threadIdx.x) * kRanks;
  const unsigned long long qend = min(total, q + kRanks);
  while (q < qend) {
    int d = pb.r;
    unsigned long long base = 0;
    while (d >= 1 && q >= base + pb.lvl_total[d - 1]) {
      base += pb.lvl_total[d - 1];
      --d;
    }
    if (d < 1) break;
    const int m = 2 * d - 1;
    const unsigned long long l0 = q - base;
    const unsigned long long l1 = min(qend - base, pb.lvl_total[d - 1]);
    int I[kEnumMaxRows];
    unrank(l0, N, m, I);
    for (unsigned long long lr = l0; lr < l1; ++lr) {
      if (lr > l0) next_comb(N, m, I);
      if (!valid_set(I, m, tb.BK)) continue;
      double H[kEnumMaxRows * 2 * kEnumMaxD];
      build_rows(va, pb.r, d, I, m, tb, H);
      double ct[2 * kEnumMaxD];
      if (!null_vector_fp64<kEnumMaxRows>(H, m, ct)) continue;
      eval_vertex(va, n, pb.r, d, I, m, ct, +1, tb, best, lr, -1, nullptr, nullptr, status);
      eval_vertex(va, n, pb.r, d, I, m, ct, -1, tb, best, lr, -1, nullptr, nullptr, status);
    }
    q = base + l1;
  }
  EnumBest* sb = reinterpret_cast<EnumBest*>(sh.comb);  // NT entries
  __syncthreads();
  sb[threadIdx.x] = best;
  __syncthreads();
  for (int h = NT / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h && enum_better(sb[threadIdx.x + h], sb[threadIdx.x])) sb[threadIdx.x] = sb[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) ebest[pb.eb_off + chunk] = sb[0];
  __syncthreads();
}

template <int PT>
__global__ void __launch_bounds__(kBSlots / PT, PT == 4 ? 6 : 2) batched_score_kernel(
    const BProb* __restrict__ probs, const BItem* __restrict__ items, int nitems, int* __restrict__ counter,
    const BTable* __restrict__ btab, const EnumTables* __restrict__ etab, uint64_t* __restrict__ keys,
    EnumBest* __restrict__ ebest, int32_t* status) {
  __shared__ BShared sh;
  for (;;) {
    if (threadIdx.x == 0) sh.next = atomicAdd(counter, 1);
    __syncthreads();
    const int it = sh.next;
    __syncthreads();
    if (it >= nitems) break;
    const BItem w = items[it];
    const BProb pb = probs[w.p];
    if (pb.exact) {
      b_enum_item<kBSlots / PT>(pb, etab[pb.K], w.s0, sh, ebest, status);
      continue;
    }
    const BTable& tb = btab[pb.K];
    switch (pb.r) {
      case 1: b_dispatch_k<1, PT>(pb, tb, w.s0, sh, keys); break;
      case 2: b_dispatch_k<2, PT>(pb, tb, w.s0, sh, keys); break;
      case 3: b_dispatch_k<3, PT>(pb, tb, w.s0, sh, keys); break;
      case 4: b_dispatch_k<4, PT>(pb, tb, w.s0, sh, keys); break;
      case 5: b_dispatch_k<5, PT>(pb, tb, w.s0, sh, keys); break;
      case 6: b_dispatch_k<6, PT>(pb, tb, w.s0, sh, keys); break;
      case 7: b_dispatch_k<7, PT>(pb, tb, w.s0, sh, keys); break;
      default: b_dispatch_k<8, PT>(pb, tb, w.s0, sh, keys); break;
    }
  }
}

template <int PT>
int batched_blocks_per_sm(int* blocks) {
  return cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, batched_score_kernel<PT>, kBSlots / PT, 0),
                    "occupancy query");
}

template <int PT>
void launch_batched_score(int grid, cudaStream_t st, const BProb* probs, const BItem* items, int nitems, int* counter,
                          const BTable* btab, const EnumTables* etab, uint64_t* keys, EnumBest* ebest,
                          int32_t* status) {
  batched_score_kernel<PT><<<grid, kBSlots / PT, 0, st>>>(probs, items, nitems, counter, btab, etab, keys, ebest, status);
}

#define LRQ_BATCHED_FORM(PREFIX, PT)                                                                                  \
  PREFIX template int batched_blocks_per_sm<PT>(int*);                                                                \
  PREFIX template void launch_batched_score<PT>(int, cudaStream_t, const BProb*, const BItem*, int, int*,             \
                                                const BTable*, const EnumTables*, uint64_t*, EnumBest*, int32_t*);
LRQ_BATCHED_FORM(extern, 1)
LRQ_BATCHED_FORM(extern, 4)

}  // namespace lrq
