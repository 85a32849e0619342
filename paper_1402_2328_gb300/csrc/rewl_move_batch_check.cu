// rewl_move_batch_check.cu -- move kernel of batched instances that also takes every decision in float64.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move_batch<true, false>(const State *, const int4 *, int, size_t, const MoveCfg &, cudaStream_t);

} // namespace rewl
