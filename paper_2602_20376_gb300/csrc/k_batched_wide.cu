// k_batched_wide.cu -- the batched scoring kernel with one slot a thread, for
// batches whose longest items set their time (batched_score.cuh).
#include "batched_score.cuh"

namespace lrq {

int batched_wide_blocks_per_sm(int* blocks) {
  return cuda_check(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, batched_score_kernel<1>, kBSlots, 0),
                    "occupancy query");
}

void launch_batched_wide(int grid, cudaStream_t st, const BProb* probs, const BItem* items, int nitems, int* counter,
                         const BTable* btab, const EnumTables* etab, uint64_t* keys, EnumBest* ebest, int32_t* status) {
  batched_score_kernel<1><<<grid, kBSlots, 0, st>>>(probs, items, nitems, counter, btab, etab, keys, ebest, status);
}

}  // namespace lrq
