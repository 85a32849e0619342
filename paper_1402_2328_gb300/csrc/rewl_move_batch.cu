// rewl_move_batch.cu -- move kernel of batched instances.
#include "rewl_move.cuh"

namespace rewl {

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

template cudaError_t start_move_batch<false, false>(const State *, const int4 *, int, size_t, const MoveCfg &, cudaStream_t);

} // namespace rewl
