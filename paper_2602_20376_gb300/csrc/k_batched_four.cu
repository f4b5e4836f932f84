// k_batched_four.cu -- the batched scoring kernel with four slots a thread, for
// batches that fill the chip (batched_score.cuh).
#include "batched_score.cuh"

namespace lrq {

LRQ_BATCHED_FORM(, 4)

}  // namespace lrq
