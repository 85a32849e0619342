// rewl_kernels.cu -- the REWL hot path on sm_103a.
//
//   k_move        (rewl_move.cuh) WL moves (Sec. 2): one warp per walker, lattice and ln g shadow in shared
//                 memory; up to 32 proposals are evaluated in parallel, then resolved in
//                 order (the batch ends before a proposal whose neighbourhood an earlier accepted
//                 flip touched), so the result equals the one-move-at-a-time walk exactly.
//   k_round_tail  per-walker flatness (warp-shuffle min / sum over visited bins) and window
//                 advance: average ln g over the m walkers, H = 0, ln f /= 2 (Sec. 2); replica
//                 exchange between windows (w, w+1), Eq. (1); end of the round.
//   k_init_prep   seeded lattices and the walk into the window.
//   k_stitch      joining of Sec. 3, Eq. (2).
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "rewl_device.cuh"
#include "rewl_em.cuh"
#include "rewl_kernels.cuh"
#include "rewl_move.cuh"

namespace rewl {

template <bool ISING, bool REPLAY, bool CHECK>
__global__ void __launch_bounds__(256) k_move_thread(State s, MoveCfg c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int slot = blockIdx.x * c.walkers_per_block + threadIdx.x;
    if (threadIdx.x >= c.walkers_per_block || slot >= s.nw) return;
    move_walker_thread<ISING, REPLAY, CHECK>(s, c, slot,
                                             smem + (size_t)threadIdx.x * move_smem_per_thread_walker(s.N, s.W));
}

cudaError_t launch_move_batch(const State *states, const int4 *jobs, int njobs, size_t smem, const MoveCfg &c,
                              cudaStream_t st)
{
    if (njobs <= 0) return cudaSuccess;
    if (c.check_all) return start_move_batch<true, false>(states, jobs, njobs, smem, c, st);
    if (c.ahead) return start_move_batch<false, true>(states, jobs, njobs, smem, c, st);
    return start_move_batch<false, false>(states, jobs, njobs, smem, c, st);
}

cudaError_t launch_move(const State &s, const MoveCfg &c, cudaStream_t st)
{
    if (c.layout == 1) { // one thread per walker, c.walkers_per_block walkers (threads) per CTA
        const int G = c.walkers_per_block;
        const size_t smem = (size_t)G * move_smem_per_thread_walker(s.N, s.W);
        const dim3 grid((s.nw + G - 1) / G), block((G + 31) & ~31);
        const bool ising = s.model == 0;
        cudaError_t e;
#define REWL_LAUNCH_MOVE_T(I, R, C)                                                              \
    do {                                                                                         \
        e = cudaFuncSetAttribute(k_move_thread<I, R, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                 (int)smem);                                                     \
        if (e != cudaSuccess) return e;                                                          \
        k_move_thread<I, R, C><<<grid, block, smem, st>>>(s, c);                                 \
    } while (0)
        if (ising) {
            if (c.words) REWL_LAUNCH_MOVE_T(true, true, false);
            else if (c.check_all) REWL_LAUNCH_MOVE_T(true, false, true);
            else REWL_LAUNCH_MOVE_T(true, false, false);
        } else {
            if (c.words) REWL_LAUNCH_MOVE_T(false, true, false);
            else if (c.check_all) REWL_LAUNCH_MOVE_T(false, false, true);
            else REWL_LAUNCH_MOVE_T(false, false, false);
        }
#undef REWL_LAUNCH_MOVE_T
        return cudaGetLastError();
    }
    const int G = c.walkers_per_block;
    const size_t smem = (size_t)G * move_smem_per_walker(s.N, s.W);
    const int grid = (s.nw + G - 1) / G;
    if (s.model == 0) {
        if (c.words) return start_move<true, true, false, false>(s, c, grid, smem, st);
        if (c.check_all) return start_move<true, false, true, false>(s, c, grid, smem, st);
        if (c.ahead) return start_move<true, false, false, true>(s, c, grid, smem, st);
        return start_move<true, false, false, false>(s, c, grid, smem, st);
    }
    if (c.words) return start_move<false, true, false, false>(s, c, grid, smem, st);
    if (c.check_all) return start_move<false, false, true, false>(s, c, grid, smem, st);
    if (c.ahead) return start_move<false, false, false, true>(s, c, grid, smem, st);
    return start_move<false, false, false, false>(s, c, grid, smem, st);
}

// ---------------------------------------------------------------------------------------
// Seeded lattices and prep into the window: one warp per walker, the lattice in shared memory (a
// 16-bit cell per site, the state in the low byte, a claim in the high one).  Far from the window a proposal is accepted by the sign of its
// energy change alone, so a batch of 32 has no serial part but its conflicts (a site or a neighbour
// that an earlier step of the batch changed: the batch ends there); near it a prefix sum finds the
// step that reaches the window, and that step is decided by itself.
// Bound by the latency of a batch.  Potts q=10 L=80, 1024 walkers, rewl_init with the lattices
// and bins read back: 548 ms with one thread per walker on global memory, 6.8 ms with a warp each.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ int dist_to(int k, int lo, int hi)
{
    return k < lo ? lo - k : (k > hi ? k - hi : 0);
}

// bin of the lattice in `cell` (no claims pending), by the whole warp
__device__ __forceinline__ int warp_bin(const uint16_t *cell, const Lattice &lat, bool ising, int lane)
{
    int sat = 0; // satisfied bonds, each site's to the right and down
    for (int i = lane; i < lat.N; i += 32) {
        int l, r, u, d;
        lat.nbrs(i, l, r, u, d);
        sat += (int)(cell[i] == cell[r]) + (int)(cell[i] == cell[d]);
    }
    sat = __reduce_add_sync(FULL, sat);
    return ising ? (4 * lat.N - 2 * sat) / 4 : 2 * lat.N - sat; // E = 2N - 2 sat, or -sat
}

template <bool ISING>
__global__ void __launch_bounds__(128) k_init_prep(State s, long long prep_budget)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int DM = ISING ? 2 : 4;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int slot = blockIdx.x * (blockDim.x >> 5) + wib;
    if (slot >= s.nw) return;
    const int w = slot / s.m, lo = s.lo[w], hi = s.hi[w], N = s.N;
    unsigned char *cellb = smem + (size_t)wib * prep_smem_per_walker(N);
    uint16_t *cell = reinterpret_cast<uint16_t *>(cellb);
    const Lattice lat{s.L, N, s.magic};
    const unsigned below = (1u << lane) - 1u;
    for (int c = lane; 4 * c < N; c += 32) {
        const u32x4 r = philox((uint32_t)c, 0u, (uint32_t)(s.slot0 + slot), (s.inst << 8) | TAG_INIT,
                               s.key0, s.key1);
        const uint32_t wv[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * c + j < N) {
                const int8_t v = ISING ? (int8_t)((wv[j] >> 31) ? -1 : 1) : (int8_t)mulhi(wv[j], (uint32_t)s.q);
                cell[4 * c + j] = (uint16_t)((NO_CLAIM << 8) | (uint8_t)v);
            }
    }
    __syncwarp();
    int k = warp_bin(cell, lat, ISING, lane);
    unsigned long long ps = 0;
    const unsigned long long budget = (unsigned long long)prep_budget * (unsigned long long)N;
    int restarts = 0;
    for (int phase = 0; phase < 2 && dist_to(k, lo, hi) > 0; ++phase) {
        if (phase == 1) { // restart from the ground state, or the checkerboard for an upper window
            const bool top = 2 * lo > (ISING ? N : 2 * N);
            for (int j = lane; j < N; j += 32) {
                const bool odd = top && (((j % s.L) + (j / s.L)) & 1);
                const int8_t v = ISING ? (int8_t)(odd ? -1 : 1) : (int8_t)(odd ? 1 : 0);
                cell[j] = (uint16_t)((NO_CLAIM << 8) | (uint8_t)v);
            }
            __syncwarp();
            k = top ? warp_bin(cell, lat, ISING, lane) : 0;
            ++restarts;
        }
        const unsigned long long end = ps + budget;
        // lane j's draw of step at + j; the next 32 are drawn while a batch waits for its lattice
        auto draw = [&](unsigned long long at) {
            const unsigned long long i = at + (unsigned long long)lane;
            return philox((uint32_t)i, (uint32_t)(i >> 32), (uint32_t)(s.slot0 + slot), (s.inst << 8) | TAG_PREP,
                          s.key0, s.key1);
        };
        u32x4 r = draw(ps);
        while (dist_to(k, lo, hi) > 0 && ps < end) {
            const int n = (int)min(32ULL, end - ps);
            const int site = (int)mulhi(r.x, (uint32_t)N);
            int nl, nr, nu, nd;
            lat.nbrs(site, nl, nr, nu, nd);
            // claims: the lowest lane that proposes a site marks it
            if (lane < n) cellb[2 * site + 1] = (uint8_t)lane;
            __syncwarp();
            unsigned c0 = cell[site], c1 = cell[nl], c2 = cell[nr], c3 = cell[nu], c4 = cell[nd];
            const uint32_t nbytes = __byte_perm(__byte_perm(c1, c2, 0x0040), __byte_perm(c3, c4, 0x0040), 0x5410);
            const uint32_t s0 = c0 & 0xffu;
            const u32x4 rn = draw(ps + 32ULL);
            int snew, dk;
            if (ISING) {
                snew = -(int)(int8_t)s0;
                dk = 2 - __popc(bytes_unequal<true>(nbytes, s0));
            } else {
                snew = (int)s0 + 1 + (int)mulhi(r.y, (uint32_t)(s.q - 1));
                if (snew >= s.q) snew -= s.q;
                dk = __popc(bytes_unequal<false>(nbytes, (uint32_t)snew)) - __popc(bytes_unequal<false>(nbytes, s0));
            }
            bool dup = false; // an earlier lane proposes the same site
            if (__any_sync(FULL, lane < n && (c0 >> 8) != (unsigned)lane)) {
                unsigned own = c0 >> 8;
                for (int it = 0; it < 32; ++it) { // each pass lowers some claim: ends within 32 passes
                    const bool again = lane < n && own > (unsigned)lane;
                    if (!__any_sync(FULL, again)) break;
                    if (again) cellb[2 * site + 1] = (uint8_t)lane;
                    __syncwarp();
                    own = cellb[2 * site + 1];
                    __syncwarp();
                }
                dup = lane < n && own < (unsigned)lane;
                c0 = cell[site];
                c1 = cell[nl];
                c2 = cell[nr];
                c3 = cell[nu];
                c4 = cell[nd];
            }
            const unsigned claims = (shl_clamp(1u, c0 >> 8) | shl_clamp(1u, c1 >> 8) | shl_clamp(1u, c2 >> 8) |
                                     shl_clamp(1u, c3 >> 8) | shl_clamp(1u, c4 >> 8)) & below;
            __syncwarp();
            if (lane < n) cellb[2 * site + 1] = (uint8_t)NO_CLAIM;
            // accepted while the walker stays on its side of the window.  The batch ends before a step whose
            // site or neighbour an earlier accepted step proposes, and behind an accepted step whose
            // claim an earlier lane holds (nobody else sees that one).
            const bool above = k > hi;
            bool acc = above ? dk <= 0 : dk >= 0;
            const unsigned accs = __ballot_sync(FULL, acc);
            int done = (int)__reduce_min_sync(FULL, lane >= n || (claims & accs) ? (unsigned)lane
                                                                                 : (dup && acc ? lane + 1u : 32u));
            const int d = acc && lane < done ? dk : 0;
            if (dist_to(k, lo, hi) > DM * 32) {
                k += __reduce_add_sync(FULL, d);
            } else {
                int pre = d; // inclusive prefix sum
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(FULL, pre, o);
                    if (lane >= o) pre += v;
                }
                const int kj = k + pre;
                const bool cross = lane < done && (above ? kj <= hi : kj >= lo);
                const int f = (int)__reduce_min_sync(FULL, cross ? (unsigned)lane : 32u);
                if (f < 32) { // step f reaches the window or the other side of it
                    const int kn = __shfl_sync(FULL, kj, f), kb = kn - __shfl_sync(FULL, d, f);
                    const bool accf = dist_to(kn, lo, hi) <= dist_to(kb, lo, hi);
                    k = accf ? kn : kb;
                    if (lane == f) acc = accf;
                    done = f + 1;
                } else {
                    k += __shfl_sync(FULL, pre, 31);
                }
            }
            if (lane < done && acc) cellb[2 * site] = (uint8_t)snew; // distinct sites
            ps += (unsigned long long)done;
            if (done == 32) r = rn;
            else r = draw(ps);
            __syncwarp();
        }
    }
    int8_t *sp = s.spins + (size_t)slot * s.spin_stride; // cfg[slot] == slot at start
    for (int i = lane; i < N; i += 32) sp[i] = (int8_t)(cell[i] & 0xffu);
    if (lane == 0) {
        s.k[slot] = k;
        s.cfg[slot] = slot;
        s.pstep[slot] = ps;
        s.restarts[slot] = restarts;
        if (dist_to(k, lo, hi) > 0) atomicOr(&s.status->err, ERR_PREP);
    }
}

cudaError_t launch_init_prep(const State &s, long long prep_budget, cudaStream_t st)
{
    const size_t per = prep_smem_per_walker(s.N);
    int g = 4; // walkers per CTA; the lattice of one fits whatever its size
    while (g > 1 && (size_t)g * per > MAX_SMEM_PER_CTA) g >>= 1;
    const size_t smem = (size_t)g * per;
    const int grid = (s.nw + g - 1) / g;
    cudaError_t e = s.model == 0
                        ? cudaFuncSetAttribute(k_init_prep<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                        : cudaFuncSetAttribute(k_init_prep<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (s.model == 0) k_init_prep<true><<<grid, 32 * g, smem, st>>>(s, prep_budget);
    else k_init_prep<false><<<grid, 32 * g, smem, st>>>(s, prep_budget);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// The rest of a round after the moves, in one launch: flatness and window advance (one CTA per
// window), replica exchange (by whichever CTA of a window pair comes second), end of the round (by
// the last CTA).  No CTA waits for another: each passes an arrival counter and goes on or leaves.
// As three launches (13 + 8 + 3 us and the gaps between them) this took 19 us of a round of Ising
// L=64 32 x 16, as one 11 us; what is left is launch latency and chains of dependent L2 loads.
// ---------------------------------------------------------------------------------------

// Flatness + window advance (Sec. 2).
__device__ __forceinline__ void check_window(const State &s, const int w, const double flatness,
                                             const double lnf_final)
{
    if (s.status->done || s.finished[w]) return;
    const int m = s.m, W = s.W, nb = s.hi[w] - s.lo[w] + 1;
    uint8_t *mask = s.mask + (size_t)w * W;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        if (mask[b]) continue;
        uint32_t any = 0u; // the m loads are independent, so they overlap
#pragma unroll 8
        for (int i = 0; i < m; ++i) any |= s.H[(size_t)(w * m + i) * W + b];
        if (any) mask[b] = 1;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    // visited bins of the window (for t of the 1/t schedule)
    __shared__ int nvis_w[32];
    int nv = 0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) nv += mask[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nv += __shfl_xor_sync(FULL, nv, o);
    if (lane == 0) nvis_w[wid] = nv;
    const bool tmode = s.mode[w] != 0;
    __shared__ int notflat; // walkers of the window not (yet) flat
    if (threadIdx.x == 0) notflat = 0;
    __syncthreads();
    for (int i = wid; i < m && !tmode; i += nwarp) {
        const int g = w * m + i;
        if (s.flat[g]) continue;
        const uint32_t *H = s.H + (size_t)g * W;
        unsigned long long sum = 0;
        uint32_t mn = 0xffffffffu;
        int cnt = 0;
#pragma unroll 8
        for (int b = lane; b < nb; b += 32) { // both loads unconditional: they overlap
            const uint32_t v = H[b];
            if (mask[b]) {
                sum += v;
                mn = min(mn, v);
                ++cnt;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sum += __shfl_xor_sync(FULL, sum, o);
            mn = min(mn, __shfl_xor_sync(FULL, mn, o));
            cnt += __shfl_xor_sync(FULL, cnt, o);
        }
        if (lane == 0) {
            if (cnt > 0 && __dmul_rn((double)mn, (double)cnt) >= __dmul_rn(flatness, (double)sum))
                s.flat[g] = 1;
            else
                atomicAdd(&notflat, 1);
        }
    }
    __syncthreads();
    if (notflat != 0) return; // 1/t mode: every check averages and sets ln f = 1/t
    // ln f after this advance (every thread computes the same value)
    long long nvis = 0;
    for (int i = 0; i < nwarp; ++i) nvis += nvis_w[i];
    // 1/t with t = moves per walker / visited bins, i.e. ln f = visited bins / moves
    const double inv_t = nvis > 0 ? __ddiv_rn((double)nvis, (double)s.step[w * m]) : 0.0;
    bool to_t = false;
    double nl;
    if (tmode) {
        nl = inv_t;
    } else {
        nl = __dmul_rn(s.lnf[w], 0.5);
        if (s.schedule == 1 && nl < inv_t) {
            to_t = true;
            nl = inv_t;
        }
    }
    // a window about to finish keeps its walkers' last fragments (resampling error bars, Sec. 3)
    const bool finishing = nl < lnf_final;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        double acc = 0.0;
        for (int i = 0; i < m; ++i) acc = __dadd_rn(acc, s.lng[(size_t)(w * m + i) * W + b]);
        const double avg = __ddiv_rn(acc, (double)m);
        for (int i = 0; i < m; ++i) {
            if (finishing) s.frag[(size_t)(w * m + i) * W + b] = s.lng[(size_t)(w * m + i) * W + b];
            s.lng[(size_t)(w * m + i) * W + b] = avg;
            s.H[(size_t)(w * m + i) * W + b] = 0u;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 0; i < m; ++i) s.flat[w * m + i] = 0;
        if (to_t) s.mode[w] = 1;
        s.lnf[w] = nl;
        if (s.iter[w] == 0) s.it1_round[w] = s.status->round + 1;
        s.iter[w] += 1;
        if (finishing) s.finished[w] = 1;
    }
}

// Partner permutation of the exchange of pair (gw, gw+1) in round rd (global window index gw):
// Fisher-Yates from Philox draws (i, rd, gw, swap tag), i = m-1 .. 1.  One warp; perm in shared
// memory, valid after the call for every lane.
__device__ __forceinline__ void exchange_perm(const State &s, int gw, long long rd, int *perm, int *draw)
{
    const int lane = threadIdx.x & 31, m = s.m;
    const uint32_t tag = (s.inst << 8) | TAG_SWAP;
    for (int i = lane; i < m; i += 32) {
        perm[i] = i;
        if (i >= 1) {
            const u32x4 r = philox((uint32_t)i, (uint32_t)rd, (uint32_t)gw, tag, s.key0, s.key1);
            draw[i] = (int)mulhi(r.x, (uint32_t)(i + 1));
        }
    }
    __syncwarp();
    if (lane == 0)
        for (int i = m - 1; i >= 1; --i) {
            const int j = draw[i];
            const int t = perm[i];
            perm[i] = perm[j];
            perm[j] = t;
        }
    __syncwarp();
}

// Accept decision of Eq. (1) for partner pair i: ln P >= 0 or ln u < ln P, u from Philox
// (m + i, rd, gw, swap tag).
__device__ __forceinline__ bool exchange_accept(const State &s, int gw, long long rd, int i, double lnP)
{
    if (lnP >= 0.0) return true;
    const u32x4 r = philox((uint32_t)(s.m + i), (uint32_t)rd, (uint32_t)gw, (s.inst << 8) | TAG_SWAP,
                           s.key0, s.key1);
    return lnu64(r.x) < lnP;
}

// Replica exchange (Eq. 1) of windows (w, w+1), w of the parity of round rd, by one warp: configuration
// indices and bins change places.  The permutation's random draws and the m decisions are lane-parallel
// (each decision touches its own two walker slots); only the Fisher-Yates swaps themselves run in order.
// Other CTAs of the launch wrote some of what is read here, so loads go past the L1.
__device__ __forceinline__ void swap_windows(const State &s, const int w, const long long rd)
{
    const int lane = threadIdx.x & 31;
    const int m = s.m, W = s.W;
    __shared__ int perm[MAX_M];
    __shared__ int draw[MAX_M];
    exchange_perm(s, s.w0 + w, rd, perm, draw);
    const int loA = s.lo[w], hiA = s.hi[w], loB = s.lo[w + 1], hiB = s.hi[w + 1];
    unsigned acc = 0;
    for (int i = lane; i < m; i += 32) {
        const int a = w * m + i, b = (w + 1) * m + perm[i];
        const int kx = __ldcg(s.k + a), ky = __ldcg(s.k + b);
        if (kx < loB || kx > hiB || ky < loA || ky > hiA) continue;
        const double *ga = s.lng + (size_t)a * W, *gb = s.lng + (size_t)b * W;
        const double lnP = __dadd_rn(__dsub_rn(__ldcg(ga + (kx - loA)), __ldcg(ga + (ky - loA))),
                                     __dsub_rn(__ldcg(gb + (ky - loB)), __ldcg(gb + (kx - loB))));
        if (exchange_accept(s, s.w0 + w, rd, i, lnP)) {
            const int t = s.cfg[a];
            s.cfg[a] = s.cfg[b];
            s.cfg[b] = t;
            s.k[a] = ky;
            s.k[b] = kx;
            ++acc;
        }
    }
    acc = __reduce_add_sync(FULL, acc);
    if (lane == 0) {
        s.swap_att[w] += (unsigned long long)m;
        s.swap_acc[w] += acc;
    }
}

// Arrival of this CTA at a counter, after everything its threads wrote: the number of CTAs that came
// before it.  What those wrote can be read after the call.
__device__ __forceinline__ unsigned arrive(unsigned *counter)
{
    __shared__ unsigned before;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        before = atomicAdd(counter, 1u);
        __threadfence();
    }
    __syncthreads();
    return before;
}

// Window w's part of the end of a round.  s.sync: one counter per pair of the round, then one for
// the windows; all zero between launches.
__device__ __forceinline__ void round_tail(const State &s, const int w, const double flatness, const double lnf_final,
                                           const bool measure)
{
    if (s.status->done) return;
    const long long rd = s.status->round;
    if (measure) // before the arrival below, after which configurations move
        for (int i = threadIdx.x >> 5; i < s.m; i += blockDim.x >> 5) measure_walker(s, w * s.m + i, w, threadIdx.x & 31);
    check_window(s, w, flatness, lnf_final);
    // pairs (a, a+1) with the global window index w0 + a of the parity of the round
    const int a = ((w + s.w0 - rd) & 1) == 0 ? w : w - 1;
    if (a >= 0 && a + 1 < s.h) {
        unsigned *counter = s.sync + (a >> 1);
        if (arrive(counter) == 1u) {
            if (threadIdx.x < 32) swap_windows(s, a, rd);
            if (threadIdx.x == 0) *counter = 0u;
        }
    }
    unsigned *counter = s.sync + (s.h + 1) / 2;
    if (arrive(counter) != (unsigned)s.h - 1u) return;
    int open = s.production;
    for (int i = threadIdx.x; i < s.h; i += blockDim.x) open |= !__ldcg(s.finished + i);
    const bool all = !__syncthreads_or(open);
    if (threadIdx.x == 0) {
        *counter = 0u;
        s.status->round = rd + 1;
        if (all) s.status->done = 1;
    }
}

__global__ void __launch_bounds__(512) k_round_tail(State s, double flatness, double lnf_final)
{
    round_tail(s, blockIdx.x, flatness, lnf_final, measured_in_tail(s));
}

// tab[b] = (instance, window); prm[instance] = (flatness, ln f_final)
__global__ void __launch_bounds__(512) k_round_tail_batch(const State *__restrict__ states,
                                                          const int2 *__restrict__ tab,
                                                          const double2 *__restrict__ prm)
{
    const int2 t = tab[blockIdx.x];
    const State s = states[t.x];
    const double2 p = prm[t.x];
    round_tail(s, t.y, p.x, p.y, false);
}

cudaError_t launch_round_tail_batch(const State *states, const int2 *tab, int n, const double2 *prm,
                                    cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_round_tail_batch<<<n, 512, 0, st>>>(states, tab, prm);
    return cudaGetLastError();
}

cudaError_t launch_round_tail(const State &s, double flatness, double lnf_final, cudaStream_t st)
{
    k_round_tail<<<s.h, 512, 0, st>>>(s, flatness, lnf_final);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Window-sharded runs: the exchange of the pair that straddles a shard boundary (Eq. 1).
// Each shard runs its windows' rounds as usual; for the pair (gw, gw+1) across the boundary,
// the shard of gw (side 1, its last window) and the shard of gw+1 (side 0, its first window)
// trade, after the round, their walkers' bins, their half of ln P, and the lattices of the
// accepted pairs.  Both sides draw the same permutation and the same random numbers, and add
// the halves in the same order as the single-device exchange, so every decision is the same.
// The round whose exchange this is has just ended: rd = round counter - 1.  One warp each.
// ---------------------------------------------------------------------------------------
struct BndPair {
    int lw, gw;   // local window on this side, global index of the pair's lower window
    long long rd; // round of the exchange
    bool active;  // the pair exchanges in this round
};

__device__ __forceinline__ BndPair bnd_pair(const State &s, int side)
{
    BndPair b;
    b.lw = side ? s.h - 1 : 0;
    b.gw = side ? s.w0 + s.h - 1 : s.w0 - 1;
    b.rd = s.status->round - 1;
    b.active = b.rd >= 0 && ((b.rd - b.gw) & 1) == 0;
    return b;
}

__global__ void k_bnd_bins(State s, int side, int *bins)
{
    const int lw = side ? s.h - 1 : 0;
    for (int i = threadIdx.x; i < s.m; i += blockDim.x) bins[i] = s.k[lw * s.m + i];
}

__global__ void k_bnd_half(State s, int side, int plo, int phi, const int *pbins, double *half)
{
    __shared__ int perm[MAX_M];
    __shared__ int draw[MAX_M];
    const BndPair b = bnd_pair(s, side);
    const int lane = threadIdx.x & 31, m = s.m;
    if (!b.active) {
        for (int i = lane; i < m; i += 32) half[i] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    exchange_perm(s, b.gw, b.rd, perm, draw);
    const int lo = s.lo[b.lw], hi = s.hi[b.lw];
    for (int i = lane; i < m; i += 32) {
        double v = __longlong_as_double(0x7ff8000000000000LL); // NaN: the pair cannot exchange
        if (side) { // own walker i of the lower window holds X
            const int a = b.lw * m + i;
            const int kx = s.k[a], ky = pbins[perm[i]];
            const double *g = s.lng + (size_t)a * s.W;
            if (kx >= plo && kx <= phi && ky >= lo && ky <= hi) v = __dsub_rn(g[kx - lo], g[ky - lo]);
        } else { // own walker perm[i] of the upper window holds Y
            const int a = b.lw * m + perm[i];
            const int kx = pbins[i], ky = s.k[a];
            const double *g = s.lng + (size_t)a * s.W;
            if (kx >= lo && kx <= hi && ky >= plo && ky <= phi) v = __dsub_rn(g[ky - lo], g[kx - lo]);
        }
        half[i] = v;
    }
}

__global__ void k_bnd_decide(State s, int side, const double *half, const double *phalf, uint8_t *acc,
                             int8_t *lat_out)
{
    __shared__ int perm[MAX_M];
    __shared__ int draw[MAX_M];
    const BndPair b = bnd_pair(s, side);
    const int lane = threadIdx.x & 31, m = s.m;
    if (!b.active) {
        for (int i = lane; i < m; i += 32) acc[i] = 0;
        return;
    }
    exchange_perm(s, b.gw, b.rd, perm, draw);
    unsigned na = 0;
    for (int i = lane; i < m; i += 32) {
        const double lower = side ? half[i] : phalf[i], upper = side ? phalf[i] : half[i];
        const bool ok = lower == lower && upper == upper &&
                        exchange_accept(s, b.gw, b.rd, i, __dadd_rn(lower, upper));
        acc[i] = ok ? 1 : 0;
        na += ok;
    }
    na = __reduce_add_sync(FULL, na);
    __syncwarp();
    // the lattices this side hands over (read before the partner's arrive)
    for (int i = 0; i < m; ++i) {
        if (!acc[i]) continue;
        const int slot = b.lw * m + (side ? i : perm[i]);
        const int8_t *src = s.spins + (size_t)s.cfg[slot] * s.spin_stride;
        for (int j = lane; j < s.N; j += 32) lat_out[(size_t)i * s.N + j] = src[j];
    }
    if (side && lane == 0) { // the counters of pair gw live with its lower window
        s.swap_att[b.lw] += (unsigned long long)m;
        s.swap_acc[b.lw] += na;
    }
}

__global__ void k_bnd_import(State s, int side, const int *pbins, const uint8_t *acc, const int8_t *plat)
{
    __shared__ int perm[MAX_M];
    __shared__ int draw[MAX_M];
    const BndPair b = bnd_pair(s, side);
    const int lane = threadIdx.x & 31, m = s.m;
    if (!b.active) return;
    exchange_perm(s, b.gw, b.rd, perm, draw);
    for (int i = 0; i < m; ++i) {
        if (!acc[i]) continue;
        const int slot = b.lw * m + (side ? i : perm[i]);
        int8_t *dst = s.spins + (size_t)s.cfg[slot] * s.spin_stride;
        for (int j = lane; j < s.N; j += 32) dst[j] = plat[(size_t)i * s.N + j];
        if (lane == 0) s.k[slot] = side ? pbins[perm[i]] : pbins[i];
    }
}

cudaError_t launch_bnd_bins(const State &s, int side, int *bins, cudaStream_t st)
{
    k_bnd_bins<<<1, 128, 0, st>>>(s, side, bins);
    return cudaGetLastError();
}

cudaError_t launch_bnd_half(const State &s, int side, int plo, int phi, const int *pbins, double *half,
                            cudaStream_t st)
{
    k_bnd_half<<<1, 32, 0, st>>>(s, side, plo, phi, pbins, half);
    return cudaGetLastError();
}

cudaError_t launch_bnd_decide(const State &s, int side, const double *half, const double *phalf,
                              uint8_t *acc, int8_t *lat_out, cudaStream_t st)
{
    k_bnd_decide<<<1, 32, 0, st>>>(s, side, half, phalf, acc, lat_out);
    return cudaGetLastError();
}

cudaError_t launch_bnd_import(const State &s, int side, const int *pbins, const uint8_t *acc,
                              const int8_t *plat, cudaStream_t st)
{
    k_bnd_import<<<1, 32, 0, st>>>(s, side, pbins, acc, plat);
    return cudaGetLastError();
}

__global__ void k_set_done(State s)
{
    int all = !s.production;
    for (int w = 0; w < s.h; ++w) all &= s.finished[w];
    s.status->done = all;
}

cudaError_t launch_set_done(const State &s, cudaStream_t st)
{
    k_set_done<<<1, 1, 0, st>>>(s);
    return cudaGetLastError();
}

// Lattices in slot order from slot `first` on, one CTA per slot.
__global__ void k_gather_spins(State s, int first, int8_t *out)
{
    const int8_t *src = s.spins + (size_t)s.cfg[first + (int)blockIdx.x] * s.spin_stride;
    int8_t *dst = out + (size_t)blockIdx.x * s.N;
    if (s.vec_spins) { // N a multiple of 16
        for (int i = threadIdx.x; i < s.N >> 4; i += blockDim.x)
            reinterpret_cast<int4 *>(dst)[i] = reinterpret_cast<const int4 *>(src)[i];
    } else {
        for (int i = threadIdx.x; i < s.N; i += blockDim.x) dst[i] = src[i];
    }
}

cudaError_t launch_gather_spins(const State &s, int first, int n, int8_t *out, cudaStream_t st)
{
    k_gather_spins<<<n, 128, 0, st>>>(s, first, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Joining (Sec. 3, Eq. 2).
// ---------------------------------------------------------------------------------------
__global__ void k_window_mean(State s, double *out)
{
    const int w = blockIdx.x, nb = s.hi[w] - s.lo[w] + 1;
    for (int b = threadIdx.x; b < s.W; b += blockDim.x) {
        double v = 0.0;
        if (b < nb) {
            double acc = 0.0;
            for (int i = 0; i < s.m; ++i) acc = __dadd_rn(acc, s.lng[(size_t)(w * s.m + i) * s.W + b]);
            v = __ddiv_rn(acc, (double)s.m);
        }
        out[(size_t)w * s.W + b] = v;
    }
}

cudaError_t launch_window_mean(const State &s, double *out, cudaStream_t st)
{
    k_window_mean<<<s.h, 256, 0, st>>>(s, out);
    return cudaGetLastError();
}

// beta by the 5-point (npts 5) or 3-point stencil at window-local bin b; 0 if not defined.
__device__ int stencil_beta(const double *l, const uint8_t *v, int nb, int b, int step, int npts,
                            double de, double *beta)
{
    if (npts == 5) {
        if (b - 2 * step < 0 || b + 2 * step >= nb) return 0;
        if (!(v[b - 2 * step] && v[b - step] && v[b + step] && v[b + 2 * step])) return 0;
        const double num = __dadd_rn(
            __dsub_rn(__dadd_rn(-l[b + 2 * step], __dmul_rn(8.0, l[b + step])),
                      __dmul_rn(8.0, l[b - step])),
            l[b - 2 * step]);
        *beta = __ddiv_rn(num, __dmul_rn(__dmul_rn(12.0, de), (double)step));
        return 1;
    }
    if (b - step < 0 || b + step >= nb) return 0;
    if (!(v[b - step] && v[b + step])) return 0;
    *beta = __ddiv_rn(__dsub_rn(l[b + step], l[b - step]),
                      __dmul_rn(__dmul_rn(2.0, de), (double)step));
    return 1;
}

// Block-wide argmin of (value, key): smaller value, ties -> smaller key.
__device__ void block_argmin(double &v, int &key)
{
    __shared__ double sv[32];
    __shared__ int sk[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(FULL, v, o);
        const int ok = __shfl_xor_sync(FULL, key, o);
        if (ov < v || (ov == v && ok < key)) {
            v = ov;
            key = ok;
        }
    }
    if (lane == 0) {
        sv[wid] = v;
        sk[wid] = key;
    }
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        v = lane < nw ? sv[lane] : INFINITY;
        key = lane < nw ? sk[lane] : 0x7fffffff;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(FULL, v, o);
            const int ok = __shfl_xor_sync(FULL, key, o);
            if (ov < v || (ov == v && ok < key)) {
                v = ov;
                key = ok;
            }
        }
        if (lane == 0) {
            sv[0] = v;
            sk[0] = key;
        }
    }
    __syncthreads();
    v = sv[0];
    key = sk[0];
    __syncthreads();
}

__device__ double block_reduce_max(double v)
{
    __shared__ double sv[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = warp_max(v);
    if (lane == 0) sv[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < (int)(blockDim.x >> 5) ? sv[lane] : -INFINITY;
        v = warp_max(v);
        if (lane == 0) sv[0] = v;
    }
    __syncthreads();
    v = sv[0];
    __syncthreads();
    return v;
}

__device__ double block_reduce_sum(double v)
{
    __shared__ double sv[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if (lane == 0) sv[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < (int)(blockDim.x >> 5) ? sv[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        if (lane == 0) sv[0] = v;
    }
    __syncthreads();
    v = sv[0];
    __syncthreads();
    return v;
}

// Join bin of windows (w, w+1) behind bin `prev`, by the whole CTA: argmin |beta_w - beta_(w+1)| by the
// 5-point stencil, else the 3-point one, else the bin valid in both nearest the overlap's midpoint;
// ties -> smaller bin; -1: none.
__device__ int join_bin(const State &s, const double *mean, int w, int prev, double de, int step)
{
    const int W = s.W, first = threadIdx.x, by = blockDim.x;
    const double *la = mean + (size_t)w * W, *lb = mean + (size_t)(w + 1) * W;
    const uint8_t *va = s.mask + (size_t)w * W, *vb = s.mask + (size_t)(w + 1) * W;
    const int loa = s.lo[w], hia = s.hi[w], lob = s.lo[w + 1], hib = s.hi[w + 1];
    const int nba = hia - loa + 1, nbb = hib - lob + 1;
    for (int npts = 5; npts >= 3; npts -= 2) {
        double best = INFINITY;
        int bk = 0x7fffffff;
        for (int k = max(lob, prev + 1) + first; k <= hia; k += by) {
            if (!va[k - loa] || !vb[k - lob]) continue;
            double ba, bb;
            if (!stencil_beta(la, va, nba, k - loa, step, npts, de, &ba)) continue;
            if (!stencil_beta(lb, vb, nbb, k - lob, step, npts, de, &bb)) continue;
            const double db = fabs(__dsub_rn(ba, bb));
            if (db < best || (db == best && k < bk)) {
                best = db;
                bk = k;
            }
        }
        block_argmin(best, bk);
        if (best < INFINITY) return bk;
    }
    double bd = INFINITY;
    int bk = 0x7fffffff;
    for (int k = max(lob, prev + 1) + first; k <= hia; k += by) {
        if (!va[k - loa] || !vb[k - lob]) continue;
        const double d = fabs((double)(2 * k - (lob + hia)));
        if (d < bd || (d == bd && k < bk)) {
            bd = d;
            bk = k;
        }
    }
    block_argmin(bd, bk);
    return bd < INFINITY ? bk : -1;
}

// Joining n sets of window means (set r at mean + r h W): k_join_bins, one CTA per pair and set, finds each
// pair's best join bin as if the pair were alone; k_stitch, one CTA per set, searches a pair again, in
// order, where that bin does not lie behind the join before it, which gives the same bins as joining pair
// by pair, adds the shifts up in order, and gives every bin its value from the last window joined at or
// below it.
// Bound by float64 (2 FMA per cycle and SM) and latency, so the pairs are spread over the SMs, four
// warps each (one: 30 us, four: 12), the norm takes no exponential that cannot reach its last bit, and its
// logarithm is one thread's.  Ising L=64, 32 windows, with the copies to the host: 212 us with one CTA going
// from pair to pair, 91 us; the jackknife's 16 resamples 3000 us one after the other, 131 us at once.
// k_stitch has 256 threads: with 1024 of 64 registers each, a search again and the passes over all bins
// took longer (Ising L=16 8 x 8 89 us, now 74; Potts L=40 64 x 4 138, now 115).
// A few small windows are searched by k_stitch alone (join_alone): the launch of k_join_bins and the searches
// again, which noisy windows need more of, cost as much as they save.  us, alone / by k_join_bins: Ising L=8
// 2 x 4 50 / 53, Ising L=16 4 x 32 62 / 65, 8 x 8 75 / 78, but 78 / 65 with 8 windows of 292 bins and
// 163 / 76 with 32 of 118.
constexpr int JOIN_THREADS = 128, STITCH_THREADS = 256;
__host__ __device__ inline bool join_alone(const State &s) { return s.h <= 2 || (s.h <= 8 && s.W <= 192); }

__global__ void __launch_bounds__(JOIN_THREADS) k_join_bins(State s, const double *mean_all, double de, int step, int *joins_all,
                                                  double *at_all)
{
    const int w = blockIdx.x, r = blockIdx.y;
    const double *mean = mean_all + (size_t)r * s.h * s.W;
    const int kj = join_bin(s, mean, w, -1, de, step);
    if (threadIdx.x == 0) {
        double *at = at_all + 2 * ((size_t)r * s.h + w); // ln g of both windows at the join
        joins_all[(size_t)r * s.h + w] = kj;
        at[0] = kj >= 0 ? mean[(size_t)w * s.W + (kj - s.lo[w])] : 0.0;
        at[1] = kj >= 0 ? mean[(size_t)(w + 1) * s.W + (kj - s.lo[w + 1])] : 0.0;
    }
}

// out + r (B+1): joined ln g of set r; joins, at and ok: [n][h], [n][h][2], [n], the first two as k_join_bins left
// them unless join_alone; at becomes the windows' shifts.
__global__ void __launch_bounds__(STITCH_THREADS)
    k_stitch(State s, const double *mean_all, double de, int step, int norm, double target, double *out_all,
             int *joins_all, double *at_all, int *ok_all, int B)
{
    const int W = s.W, h = s.h;
    const double *mean = mean_all + (size_t)blockIdx.x * h * W;
    double *out = out_all + (size_t)blockIdx.x * (B + 1), *at = at_all + 2 * (size_t)blockIdx.x * h;
    int *joins = joins_all + (size_t)blockIdx.x * h, *ok = ok_all + blockIdx.x;
    __shared__ int redo, fail_s;
    __shared__ double sh_s;
    __shared__ double2 step_s[STITCH_THREADS];
    if (threadIdx.x == 0) {
        fail_s = 0;
        sh_s = 0.0;
    }
    if (join_alone(s)) // no pair has a join yet
        for (int w = threadIdx.x; w + 1 < h; w += blockDim.x) joins[w] = -1;
    __syncthreads();
    for (int w0 = 0;;) { // the first pair from w0 on whose join is not behind the one before
        if (threadIdx.x == 0) redo = h - 1;
        __syncthreads();
        for (int w = w0 + (int)threadIdx.x; w + 1 < h; w += blockDim.x)
            if (joins[w] <= (w > 0 ? joins[w - 1] : -1)) atomicMin(&redo, w);
        __syncthreads();
        const int w = redo;
        __syncthreads();
        if (w + 1 >= h) break;
        const int kj = join_bin(s, mean, w, w > 0 ? joins[w - 1] : -1, de, step);
        if (threadIdx.x == 0) {
            joins[w] = kj;
            if (kj < 0) {
                fail_s = 1;
            } else {
                at[2 * w] = mean[(size_t)w * W + (kj - s.lo[w])];
                at[2 * w + 1] = mean[(size_t)(w + 1) * W + (kj - s.lo[w + 1])];
            }
        }
        __syncthreads();
        if (fail_s) break;
        w0 = w + 1;
    }
    if (fail_s) {
        if (threadIdx.x == 0) *ok = 0;
        return;
    }
    for (int w0 = 0; w0 + 1 < h; w0 += blockDim.x) { // the chain of shifts; at[w] = shift of window w+1
        const int n = min((int)blockDim.x, h - 1 - w0), i = threadIdx.x;
        if (i < n) step_s[i] = reinterpret_cast<const double2 *>(at)[w0 + i];
        __syncthreads();
        if (i == 0) {
            double sh = sh_s;
            for (int k = 0; k < n; ++k) {
                sh = __dsub_rn(__dadd_rn(step_s[k].x, sh), step_s[k].y);
                step_s[k].x = sh;
            }
            sh_s = sh;
        }
        __syncthreads();
        if (i < n) at[w0 + i] = step_s[i].x; // behind what the next pass reads
        __syncthreads();
    }
    const double *shift = at - 1;
    for (int b = threadIdx.x; b <= B; b += blockDim.x) {
        int a = 0, z = h - 1; // windows joined at or below b: joins[0 .. a-1] <= b
        while (a < z) {
            const int mid = (a + z + 1) / 2;
            if (joins[mid - 1] <= b) a = mid;
            else z = mid - 1;
        }
        const int i = b - s.lo[a];
        double v = -INFINITY;
        if (i >= 0 && b <= s.hi[a] && s.mask[(size_t)a * W + i])
            v = a ? __dadd_rn(mean[(size_t)a * W + i], shift[a]) : mean[i];
        out[b] = v;
    }
    __syncthreads();
    if (norm == 0) {
        double mx = -INFINITY;
        for (int b = threadIdx.x; b <= B; b += blockDim.x) mx = fmax(mx, out[b]);
        mx = block_reduce_max(mx);
        double sum = 0.0;
        for (int b = threadIdx.x; b <= B; b += blockDim.x) // e^-80 of the largest term: no bit of the sum
            if (out[b] - mx > -80.0) sum += exp(out[b] - mx);
        sum = block_reduce_sum(sum);
        if (threadIdx.x == 0) sh_s = (mx + log(sum)) - target; // by one thread: a logarithm of every thread takes 5 us
        __syncthreads();
        const double cst = sh_s;
        for (int b = threadIdx.x; b <= B; b += blockDim.x)
            if (out[b] > -INFINITY) out[b] -= cst;
    } else {
        int b0 = 0x7fffffff;
        double dummy = 0.0;
        for (int b = threadIdx.x; b <= B; b += blockDim.x)
            if (out[b] > -INFINITY && b < b0) b0 = b;
        block_argmin(dummy, b0);
        if (b0 > B) {
            if (threadIdx.x == 0) *ok = 0;
            return;
        }
        const double cst = __dsub_rn(out[b0], target);
        __syncthreads();
        for (int b = threadIdx.x; b <= B; b += blockDim.x)
            if (out[b] > -INFINITY) out[b] = __dsub_rn(out[b], cst);
    }
    if (threadIdx.x == 0) *ok = 1;
}

cudaError_t launch_stitch(const State &s, int n, const double *mean, double de, int step, int norm,
                          double target, double *out, int *joins, double *at, int *ok, int B, cudaStream_t st)
{
    if (!join_alone(s)) k_join_bins<<<dim3(s.h - 1, n), JOIN_THREADS, 0, st>>>(s, mean, de, step, joins, at);
    k_stitch<<<n, STITCH_THREADS, 0, st>>>(s, mean, de, step, norm, target, out, joins, at, ok, B);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Diagnostics.
// ---------------------------------------------------------------------------------------
__global__ void k_philox(const uint32_t *ctr, const uint32_t *key, uint32_t *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const u32x4 r = philox(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3],
                           key[2 * i], key[2 * i + 1]);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

cudaError_t launch_philox(const uint32_t *ctr, const uint32_t *key, uint32_t *out, int n,
                          cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_philox<<<(n + 255) / 256, 256, 0, st>>>(ctr, key, out, n);
    return cudaGetLastError();
}

__global__ void k_lnu(const uint32_t *w, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = lnu64(w[i]);
}

cudaError_t launch_lnu(const uint32_t *w, double *out, int n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_lnu<<<(n + 255) / 256, 256, 0, st>>>(w, out, n);
    return cudaGetLastError();
}

__device__ __forceinline__ void atomic_max_pos(double *addr, double v)
{
    // non-negative doubles order like their bit patterns
    atomicMax(reinterpret_cast<unsigned long long *>(addr), (unsigned long long)__double_as_longlong(v));
}

__global__ void k_lnu_bound(uint64_t begin, uint64_t end, double *max_err, unsigned long long *n_bad)
{
    double mx = 0.0;
    unsigned long long bad = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t x = begin + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < end; x += stride) {
        const uint32_t w = (uint32_t)x;
        const double e = lnu64(w);
        const double f = (double)lnu32(w);
        mx = fmax(mx, fabs(f - e));
        bad += (e >= 0.0);
    }
    mx = warp_max(mx);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) bad += __shfl_xor_sync(FULL, bad, o);
    if ((threadIdx.x & 31) == 0) {
        atomic_max_pos(max_err, mx);
        if (bad) atomicAdd(n_bad, bad);
    }
}

cudaError_t launch_lnu_bound(uint64_t begin, uint64_t end, double *max_err,
                             unsigned long long *n_bad, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(max_err, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(n_bad, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    if (end <= begin) return cudaSuccess;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_lnu_bound<<<sms * 8, 256, 0, st>>>(begin, end, max_err, n_bad);
    return cudaGetLastError();
}

__global__ void k_seqadd(const double *x, const double *f, const uint32_t *c, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = seqadd(x[i], f[i], c[i]);
}

cudaError_t launch_seqadd(const double *x, const double *f, const uint32_t *c, double *out,
                          int n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_seqadd<<<(n + 127) / 128, 128, 0, st>>>(x, f, c, out, n);
    return cudaGetLastError();
}

} // namespace rewl

namespace rewl {

// Sums of a and b over the CTA, added in the order of block_reduce_sum: a becomes its sum, b the quotient of
// theirs.  The caller has a barrier before the next call.
__device__ __forceinline__ void block_mean(double &a, double &b)
{
    __shared__ double sa[32], sb[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(FULL, a, o);
        b += __shfl_xor_sync(FULL, b, o);
    }
    if (lane == 0) {
        sa[wid] = a;
        sb[wid] = b;
    }
    __syncthreads();
    if (wid == 0) {
        a = lane < (int)(blockDim.x >> 5) ? sa[lane] : 0.0;
        b = lane < (int)(blockDim.x >> 5) ? sb[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(FULL, a, o);
            b += __shfl_xor_sync(FULL, b, o);
        }
        if (lane == 0) { // float64 quotients are taken by one thread
            sa[0] = a;
            sb[0] = b / a;
        }
    }
    __syncthreads();
    a = sa[0];
    b = sb[0];
}

// ---------------------------------------------------------------------------------------
// Canonical averages from ln g (Eqs. 6-7): one CTA per temperature; u = <E>/N,
// c = <(E - <E>)^2> / (N T^2), weights g(E) e^{-E/T} taken relative to one near their maximum.
//
// Bound by float64, of which an SM does 2 FMA per cycle, so float64 goes only where it can reach a
// result: a float32 pass finds the largest exponent and the bins within e^-82 of it (widened by a bound of
// its own rounding error); only those, a tenth of the bins, take a quotient, an exponential and the
// sums in float64.  Every bin does where float32 is too coarse to tell (large E/T), or where one bin holds
// all the weight and c is made of the rest; the largest exponents of the threads mostly tell, so that the
// selected bins are not summed for nothing first (Ising L=8, 500 frozen temperatures: 26 us before the
// selection, 32 with it, 24 told beforehand).  Four CTAs an SM: left to itself the compiler takes 48
// registers and spills (54 us).  Ising L=64, 500 temperatures: 393 us with a float64 quotient per bin in three
// passes and two exponentials, 51 us.
// ---------------------------------------------------------------------------------------
constexpr int THERMO_THREADS = 256;
constexpr int THERMO_KEEP = 8; // weights a thread keeps between the two sums

__global__ void __launch_bounds__(THERMO_THREADS, 4)
    k_thermo(const double *__restrict__ lng, int B, int model, int N, const double *__restrict__ Ts,
             double *__restrict__ U, double *__restrict__ Cv)
{
    __shared__ double keep[THERMO_KEEP * THERMO_THREADS];
    __shared__ float mx_s[32], next_s[32], big_s[32];
    __shared__ int arg_s[32];
    __shared__ double one_s; // float64 quotients are taken by one thread
    const double T = Ts[blockIdx.x];
    if (threadIdx.x == 0) one_s = 1.0 / T;
    __syncthreads();
    const double inv = one_s;
    const float invf = (float)inv;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto energy = [&](int b) { return model == 0 ? 4 * b - 2 * N : b - 2 * N; };
    auto coarse = [&](int b) { return __fmaf_rn(-(float)energy(b), invf, (float)lng[b]); };
    // ---- float32: the largest exponent, its bin, the largest of the other threads', the largest |ln g|
    float mx = -INFINITY, next = -INFINITY, big = 0.0f;
    int arg = 0;
    for (int b = threadIdx.x; b <= B; b += blockDim.x) {
        const float l = (float)lng[b], x = __fmaf_rn(-(float)energy(b), invf, l);
        if (l > -INFINITY) big = fmaxf(big, fabsf(l));
        if (x > mx) {
            mx = x;
            arg = b;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float om = __shfl_xor_sync(FULL, mx, o);
        const int oa = __shfl_xor_sync(FULL, arg, o);
        next = fmaxf(fmaxf(next, __shfl_xor_sync(FULL, next, o)), fminf(mx, om));
        if (om > mx) {
            mx = om;
            arg = oa;
        }
        big = fmaxf(big, __shfl_xor_sync(FULL, big, o));
    }
    if (lane == 0) {
        mx_s[wid] = mx;
        next_s[wid] = next;
        big_s[wid] = big;
        arg_s[wid] = arg;
    }
    __syncthreads();
    for (int i = 0; i < THERMO_THREADS / 32; ++i) { // the same choice in every thread
        next = i == 0 ? next_s[0] : fmaxf(fmaxf(next, next_s[i]), fminf(mx, mx_s[i]));
        if (i == 0 || mx_s[i] > mx) {
            mx = mx_s[i];
            arg = arg_s[i];
        }
        big = fmaxf(big, big_s[i]);
    }
    // |coarse - exact| < 2^-22 (2N / T + max |ln g|); 8 times that here
    const float slack = 0x1p-19f * (2.0f * (float)N * fabsf(invf) + big);
    const float cut = mx - 82.0f - 2.0f * slack;
    // what the bins left out can add to s2 stays below its last bit where s2 >= enough s0
    const double enough = 1e17 * 2.5e-36 * (double)(B + 1) * 16.0 * (double)N * (double)N;
    // Where no bin beside the one of the largest exponent comes near it, the others will not reach `enough`, and
    // every bin is taken at once.  Either way is right: s2 below tells.
    const bool frozen = mx - next > 43.0f - __logf((float)(B + 1) * (float)N * (float)N);
    double s0, e1, s2, E0; // e1: mean energy from E0
    for (bool all = frozen || !(slack < 8.0f && fabs(T) < INFINITY);; all = true) {
        // every bin: energies from the bin of the largest exponent, so that a mean next to it keeps all its
        // digits, as c of a frozen lattice is a sum over the other bins
        const int e0 = all ? energy(arg) : 0;
        E0 = (double)e0;
        auto rel = [&](int b) { return (double)(energy(b) - e0); };
        auto exponent = [&](double R) { // of the bin at energy E0 + R, its ln g aside
            if (all) return (E0 + R) / T;
            const double q = R * inv; // E / T: one correction of E * (1 / T)
            return __fma_rn(__fma_rn(-q, T, R), inv, q);
        };
        double ref;
        if (all) {
            ref = -INFINITY;
            for (int b = threadIdx.x; b <= B; b += blockDim.x)
                if (lng[b] > -INFINITY) ref = fmax(ref, lng[b] - exponent(rel(b)));
            ref = block_reduce_max(ref);
        } else {
            ref = lng[arg] - exponent(rel(arg));
        }
        auto weight = [&](int b, double R) { return exp((lng[b] - exponent(R)) - ref); };
        auto counts = [&](int b) { return all ? lng[b] > -INFINITY : coarse(b) > cut; };
        s0 = e1 = 0.0;
        int n = 0;
        for (int b = threadIdx.x; b <= B; b += blockDim.x)
            if (counts(b)) {
                const double R = rel(b), w = weight(b, R);
                if (n < THERMO_KEEP) keep[n * THERMO_THREADS + threadIdx.x] = w;
                ++n;
                s0 += w;
                e1 += w * R;
            }
        block_mean(s0, e1);
        s2 = 0.0;
        n = 0;
        for (int b = threadIdx.x; b <= B; b += blockDim.x)
            if (counts(b)) {
                const double R = rel(b), de = R - e1;
                const double w = n < THERMO_KEEP ? keep[n * THERMO_THREADS + threadIdx.x] : weight(b, R);
                ++n;
                s2 += w * de * de;
            }
        s2 = block_reduce_sum(s2);
        if (all || s2 >= enough * s0) break; // else nearly one bin alone (low T): again with every bin
    }
    if (threadIdx.x == 0) {
        U[blockIdx.x] = (E0 + e1) / N;
        Cv[blockIdx.x] = s2 / s0 / ((double)N * T * T);
    }
}

cudaError_t launch_thermo(const double *lng, int model, int L, const double *T, int nT, double *U,
                          double *C, cudaStream_t st)
{
    if (nT <= 0) return cudaSuccess;
    const int N = L * L, B = model == 0 ? N : 2 * N;
    k_thermo<<<nT, THERMO_THREADS, 0, st>>>(lng, B, model, N, T, U, C);
    return cudaGetLastError();
}

} // namespace rewl

namespace rewl {

// Window means of the saved fragments leaving walker j0 + blockIdx.y out (walker order), [n][h][W].
__global__ void k_loo_mean(State s, int j0, double *out_all)
{
    const int w = blockIdx.x, j = j0 + blockIdx.y, nb = s.hi[w] - s.lo[w] + 1;
    double *out = out_all + (size_t)blockIdx.y * s.h * s.W;
    for (int b = threadIdx.x; b < s.W; b += blockDim.x) {
        double v = 0.0;
        if (b < nb) {
            double acc = 0.0;
#pragma unroll 8
            for (int i = 0; i < s.m; ++i) {
                const double x = s.frag[(size_t)(w * s.m + i) * s.W + b];
                acc = i != j ? __dadd_rn(acc, x) : acc;
            }
            v = __ddiv_rn(acc, (double)(s.m - 1));
        }
        out[(size_t)w * s.W + b] = v;
    }
}

cudaError_t launch_loo_mean(const State &s, int j0, int n, double *out, cudaStream_t st)
{
    k_loo_mean<<<dim3(s.h, n), 256, 0, st>>>(s, j0, out);
    return cudaGetLastError();
}

// err[b] = sqrt((m-1)/m sum_j (theta_j[b] - mean)^2); NaN where any theta_j is -inf.
__global__ void k_jack(const double *theta, int m, int B, double *err)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > B) return;
    double mean = 0.0;
    bool ok = true;
    for (int j = 0; j < m; ++j) {
        const double v = theta[(size_t)j * (B + 1) + b];
        ok = ok && v > -INFINITY;
        mean += v;
    }
    if (!ok) {
        err[b] = NAN;
        return;
    }
    mean /= m;
    double ss = 0.0;
    for (int j = 0; j < m; ++j) {
        const double d = theta[(size_t)j * (B + 1) + b] - mean;
        ss += d * d;
    }
    err[b] = sqrt((double)(m - 1) / m * ss);
}

cudaError_t launch_jack(const double *theta, int m, int B, double *err, cudaStream_t st)
{
    k_jack<<<(B + 64) / 64, 64, 0, st>>>(theta, m, B, err);
    return cudaGetLastError();
}

} // namespace rewl
