// rewl_move_check.cu -- move kernels that also take every decision in float64.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move<true, false, true, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);
template cudaError_t start_move<false, false, true, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);

} // namespace rewl
