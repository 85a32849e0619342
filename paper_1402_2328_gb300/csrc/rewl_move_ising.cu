// rewl_move_ising.cu -- move kernels of an Ising run.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move<true, false, false, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);
template cudaError_t start_move<true, false, false, true>(const State &, const MoveCfg &, int, size_t, cudaStream_t);

} // namespace rewl
