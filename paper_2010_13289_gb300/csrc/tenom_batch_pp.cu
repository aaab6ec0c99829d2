/* Batched stage kernels with the positivity-preserving flux limiter (Section 4.4), in a
   translation unit of their own so that they compile in parallel with the others. */
#include "tenom_batch_kernel.cuh"

namespace tenom {

StageFn pick_stage_pp(int K, int lim, int tile, bool all) {
  return all ? pick_stage_of<true, true>(K, lim, tile) : pick_stage_of<true, false>(K, lim, tile);
}

}  // namespace tenom
