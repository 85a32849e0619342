// rewl_move_replay.cu -- move kernels on caller-given random words.
#include "rewl_move_start.cuh"

namespace rewl {

template cudaError_t start_move<true, true, false, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);
template cudaError_t start_move<false, true, false, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);

} // namespace rewl
