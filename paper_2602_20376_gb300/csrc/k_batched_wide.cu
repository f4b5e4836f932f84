// k_batched_wide.cu -- the batched scoring kernel with one slot a thread, for
// batches whose longest items set their time (batched_score.cuh).
#include "batched_score.cuh"

namespace lrq {

LRQ_BATCHED_FORM(, 1)

}  // namespace lrq
