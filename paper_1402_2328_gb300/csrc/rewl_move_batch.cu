// rewl_move_batch.cu -- move kernel of batched instances.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move_batch<false, false>(const State *, const int4 *, int, size_t, const MoveCfg &, cudaStream_t);

} // namespace rewl
