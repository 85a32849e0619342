// rewl_move_start.cuh -- launches of the move kernels, for the files that instantiate them.
#pragma once
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

template <bool CHECK, bool AHEAD>
cudaError_t start_move_batch(const State *states, const int4 *jobs, int njobs, size_t smem, const MoveCfg &c,
                             cudaStream_t st)
{
    const cudaError_t e = cudaFuncSetAttribute(k_move_batch<CHECK, AHEAD>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_move_batch<CHECK, AHEAD><<<njobs, (AHEAD ? 64 : 32) * c.walkers_per_block, smem, st>>>(states, jobs, c);
    return cudaGetLastError();
}

} // namespace rewl
