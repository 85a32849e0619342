// rewl_move_potts.cu -- move kernels of a Potts run.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move<false, false, false, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);
template cudaError_t start_move<false, false, false, true>(const State &, const MoveCfg &, int, size_t, cudaStream_t);

} // namespace rewl
