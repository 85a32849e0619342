// rewl_move_check.cu -- move kernels that also take every decision in float64.
#include "rewl_move.cuh"

namespace rewl {

template <bool ISING, bool REPLAY, bool CHECK, bool AHEAD>
cudaError_t start_move(const State &s, const MoveCfg &c, int grid, size_t smem, cudaStream_t st)
{
    const cudaError_t e = cudaFuncSetAttribute(k_move<ISING, REPLAY, CHECK, AHEAD>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_move<ISING, REPLAY, CHECK, AHEAD><<<grid, (AHEAD ? 64 : 32) * c.walkers_per_block, smem, st>>>(s, c);
    return cudaGetLastError();
}

template cudaError_t start_move<true, false, true, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);
template cudaError_t start_move<false, false, true, false>(const State &, const MoveCfg &, int, size_t, cudaStream_t);

} // namespace rewl
