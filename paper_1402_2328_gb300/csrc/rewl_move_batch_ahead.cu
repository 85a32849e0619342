// rewl_move_batch_ahead.cu -- move kernel of batched instances, with a second warp per walker that draws.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move_batch<false, true>(const State *, const int4 *, int, size_t, const MoveCfg &, cudaStream_t);

} // namespace rewl
