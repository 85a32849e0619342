// rewl_em.cuh -- the (E, M) measurement of a round (Sec. 3), as its own launch or in the round's tail.
#pragma once
#include <cstdint>

#include "rewl_kernels.cuh"

namespace rewl {

// Whether the tail of a round, one CTA of 16 warps per window, takes the measurement along: up to
// two walkers a warp and 64 KB of lattices a window, which it reads in about the time of the launch
// saved; beyond that such a launch over all walkers reads them with the whole chip.  us per round of 50 moves
// and 4 windows, in the tail / on its own: Ising L=16 32 walkers 27.9 / 29.2, 64 30.3 / 30.0, 128 39.1 / 36.1;
// L=64 16 walkers (64 KB) 51.7 / 53.0, 32 55.7 / 55.5, 64 63.5 / 62.1.
__host__ __device__ inline bool measured_in_tail(const State &s)
{
    return s.hem && s.m <= 32 && (long long)s.m * s.N <= 65536;
}

// (E, M) of one walker after its moves into the histogram of its window w, by a warp: 16 spins a
// load, an up spin (+1) has its top bit clear.  Lattice rows start on 16-byte boundaries; what lies
// behind the last site is not counted.
__device__ __forceinline__ void measure_walker(const State &s, int slot, int w, int lane)
{
    const int8_t *sp = s.spins + (size_t)s.cfg[slot] * s.spin_stride;
    int up = 0;
    for (int i = lane * 16; i + 16 <= s.N; i += 512) {
        const uint4 v = *reinterpret_cast<const uint4 *>(sp + i);
        const unsigned down = ((v.x & 0x80808080u) >> 3) | ((v.y & 0x80808080u) >> 2) | ((v.z & 0x80808080u) >> 1) |
                              (v.w & 0x80808080u);
        up += 16 - __popc(down);
    }
    const int i = (s.N & ~15) + lane;
    if (i < s.N) up += sp[i] > 0;
    up = __reduce_add_sync(0xffffffffu, up);
    if (lane == 0)
        atomicAdd(&s.hem[((size_t)w * s.W + (size_t)(s.k[slot] - s.lo[w])) * (size_t)(s.N + 1) + up], 1u);
}

} // namespace rewl
