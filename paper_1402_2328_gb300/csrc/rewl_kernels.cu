// rewl_kernels.cu -- the REWL hot path on sm_103a.
//
//   k_move        WL moves (Sec. 2): one warp per walker, lattice and ln g shadow in shared
//                 memory; up to 32 proposals are evaluated in parallel, then resolved in
//                 order (the batch ends before a proposal whose neighbourhood an earlier accepted
//                 flip touched), so the result equals the one-move-at-a-time walk exactly.
//   k_check       per-walker flatness (warp-shuffle min / sum over visited bins) and window
//                 advance: average ln g over the m walkers, H = 0, ln f /= 2 (Sec. 2).
//   k_swap        replica exchange between windows (w, w+1), Eq. (1).
//   k_init_prep   seeded lattices and the walk into the window.
//   k_stitch      joining of Sec. 3, Eq. (2).
#include <cfloat>
#include <cmath>
#include <cstdint>

#include <cuda_fp16.h>

#include "rewl_device.cuh"
#include "rewl_kernels.cuh"

namespace rewl {

constexpr unsigned FULL = 0xffffffffu;

__host__ __device__ inline int pad16(int n) { return (n + 15) & ~15; }
__host__ __device__ inline int padw(int w) { return (w + 3) & ~3; }

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(FULL, v, o));
    return v;
}

// Energy change (in bins) of a proposal at `site` on lattice sp, plus the new state.
template <bool ISING>
__device__ __forceinline__ int propose_dk(const int8_t *sp, const Lattice &lat, int q, int site,
                                          int pr, int &snew)
{
    int l, r, u, d;
    lat.nbrs(site, l, r, u, d);
    const int s0 = sp[site];
    const int a0 = sp[l], a1 = sp[r], a2 = sp[u], a3 = sp[d];
    if (ISING) {
        snew = -s0;
        return (s0 * (a0 + a1 + a2 + a3)) / 2; // dE = 2 s0 sum, dk = dE / 4
    } else {
        int sn = s0 + 1 + pr;
        if (sn >= q) sn -= q;
        snew = sn;
        return (int)(s0 == a0) + (int)(s0 == a1) + (int)(s0 == a2) + (int)(s0 == a3) -
               (int)(sn == a0) - (int)(sn == a1) - (int)(sn == a2) - (int)(sn == a3);
    }
}

// ---------------------------------------------------------------------------------------
// WL moves.  Decision rule (Sec. 2): accept iff ln u < ln g(k) - ln g(k'), with the float64
// ln g the one-move-at-a-time walk would hold at that moment.
//
// One warp per walker.  Shared memory holds the lattice, an int64 shadow
// V(b) = round(ln g0(b) 2^32) + (visits) * round(ln f 2^32) of ln g over the window, and the
// proposals drawn ahead.  Moves are taken in batches of up to 32:
//   1. lane j takes the proposal of step t+j from the ring (site, neighbours, ln u: drawn
//      32 steps at a time in issue slots the walk of an earlier batch leaves idle) and evaluates
//      its energy change on the lattice as it was at the batch start;
//   2. lane x keeps the shadow of cached bin x (32 bins around the current one) in a register;
//      the cache moves when the walker nears its edge;
//   3. small ln f: lane j compares its threshold with the half-precision ratio table
//      ln g(x) - ln g(x + dk) for every cached x at once, which gives a 32-bit mask "step j is
//      surely accepted from x".  Walking the batch is then a chain of integer shifts and
//      multiply-adds on these masks, two steps at a time.  A step that is surely accepted or
//      rejected under a margin that covers every rounding and the visits since the table was
//      taken needs no more; another one is decided in float32 with those visits, and if that
//      is too close as well, in float64.
//      Large ln f, where each visit turns later decisions: the path is walked with running
//      float32 values through shuffles, every step screened by the same kind of margin;
//   4. the batch is cut before the first step that has a neighbour changed by an earlier step of
//      the batch, or shares its site with one, and behind it the side effects (spin flips, visits)
//      are applied lane-parallel.
// A step inside the float32 margin is decided from the float64 values rebuilt exactly (seqadd of
// the interval-start ln g and the visit counts); at the end of the launch the float64 ln g of
// every bin is rebuilt the same way, so the state equals that of the sequential walk bit for bit.
//
// What bounds it: the dependent chain of one batch.  A walker is one warp and the workloads have
// 1-2 walkers per SM sub-partition, so latencies set the pace, not issue slots or memory
// (measured on GB300 in cycles: integer op or FMA 4, a predicate before use 10, shuffle 24-28,
// shared load 29, ballot 23, popc 20, ffs 42, match_any of 32 different values 375).
// Ising L=64, 32 x 16, ln f = 2^-20, ms per round: 0.64 with the 32-step chain of shuffles and
// predicates before, 0.35 with the masks.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ double shadow_error(double maxabs, int T, double lnf, bool frozen)
{
    // bound on |V(b) 2^-32 - ln g(b)| in units of 2^-32 over a launch of T moves
    const long long fb = __double_as_longlong(lnf);
    const bool dyadic = (fb & 0x000fffffffffffffLL) == 0 && lnf >= 0x1p-32;
    const double M = maxabs + (double)T * lnf;
    const int ex = (int)((__double_as_longlong(M) >> 52) & 0x7ff);
    const double ulpM = ex > 52 ? __longlong_as_double((long long)(ex - 52) << 52) : 0x1p-1022;
    if (frozen) return 0.5;
    if (dyadic) return 0.5 + 64.0 * ulpM * 0x1p32; // exact additions except binade crossings
    return 0.5 + 0.5 * (double)T + (double)T * ulpM * 0x1p31; // every addition may round
}

__device__ __forceinline__ float ulpf(float x)
{
    // unit in the last place of |x| (x normal), as a power of two
    const int e = (__float_as_int(fabsf(x)) >> 23) & 0xff;
    return e > 23 ? __int_as_float((e - 23) << 23) : 0x1p-126f;
}

__device__ __forceinline__ float warp_maxf(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}

// visits of bin b since the launch started: the shadow grew by lnfq per visit
__device__ __forceinline__ uint32_t visits(const long long *V, const double *glng, int b, long long lnfq)
{
    return (uint32_t)((V[b] - __double2ll_rn(__dmul_rn(glng[b], 0x1p32))) / lnfq);
}

// Float64 decision from the exact values (rare): ln g of bins k and k' rebuilt by seqadd from
// the launch-start values and the visits recorded in the shadow.
__device__ __noinline__ bool exact_value_decision(const double *glng, const long long *V, int lo,
                                                  int k, int kp, double lnf, long long lnfq,
                                                  bool frozen, uint32_t w2)
{
    const uint32_t vk = frozen ? 0u : visits(V, glng, k - lo, lnfq);
    const uint32_t vkp = frozen ? 0u : visits(V, glng, kp - lo, lnfq);
    const double lk = seqadd(glng[k - lo], lnf, vk);
    const double lkp = seqadd(glng[kp - lo], lnf, vkp);
    const double d = __dsub_rn(lk, lkp);
    return (d >= 0.0) || (lnu64(w2) < d);
}

// The same, for the warp of one walker: every lane takes part after the lanes' shadow updates.
__device__ __forceinline__ bool exact_decision(const double *glng, const long long *V, int lo, int k,
                                               int kp, double lnf, long long lnfq, bool frozen,
                                               uint32_t w2)
{
    __syncwarp();
    return exact_value_decision(glng, V, lo, k, kp, lnf, lnfq, frozen, w2);
}

// ---- the lattice in the warp kernel's shared memory: one 16-bit cell per site, the state in the
// low byte and, while a batch is set up, the lane that proposes the site in the high byte
// (NO_CLAIM: none), so one load gives both.
constexpr unsigned NO_CLAIM = 0xffu;

// Ratio table: rows d = -DM .. DM of 32 half-precision differences ln g(x) - ln g(x + d) over
// the cached bins x; word w of a row holds x = w and x = w + 16.  A row is 80 bytes, so the
// 16-byte loads of eight lanes at eight different rows meet eight different bank groups.
constexpr int ROW_BYTES = 80;

__device__ __forceinline__ uint32_t shl_clamp(uint32_t v, uint32_t n)
{
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n)); // 0 for n >= 32
    return r;
}

// -1 if v is negative, else 0.  Spelled out: the compiler would make a comparison and a select of
// it, and a predicate takes 10 cycles before it can be used where a shift takes 4.
__device__ __forceinline__ int sign_mask(int v)
{
    int m;
    asm("shr.s32 %0, %1, 31;" : "=r"(m) : "r"(v));
    return m;
}

// a where mask m is -1, b where it is 0
__device__ __forceinline__ int pick(int m, int a, int b)
{
    int r;
    asm("lop3.b32 %0, %1, %2, %3, 0xca;" : "=r"(r) : "r"(m), "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ float pickf(int m, float a, float b)
{
    return __int_as_float(pick(m, __float_as_int(a), __float_as_int(b)));
}

// 0x01 in every byte of `p` that differs from byte value b (bytes below 128, or all +-1)
template <bool ISING> __device__ __forceinline__ uint32_t bytes_unequal(uint32_t p, uint32_t b)
{
    const uint32_t x = p ^ (b * 0x01010101u);
    if (ISING) return (x >> 7) & 0x01010101u; // +1 ^ -1 = 0xfe
    return ((x + 0x7f7f7f7fu) >> 7) & 0x01010101u;
}

// One walker's `c.T` moves; `base` is the walker's shared-memory block, the whole warp calls.
// NP: pairs of steps in a batch (16, or fewer for small lattices, where sites soon repeat).
template <bool ISING, bool REPLAY, bool CHECK, int NP>
__device__ __forceinline__ void move_walker_n(const State &s, const MoveCfg &c, const int slot,
                                              unsigned char *base, const int lane)
{
    constexpr int DM = ISING ? 2 : 4; // largest |bin change| of a move
    uint16_t *cell = reinterpret_cast<uint16_t *>(base);
    uint8_t *cellb = base;
    long long *V = reinterpret_cast<long long *>(base + 2 * pad16(s.N));
    uint32_t *vis = reinterpret_cast<uint32_t *>(V + padw(s.W)); // [W bits] bin visited
    unsigned char *tab = reinterpret_cast<unsigned char *>(vis + visw(s.W));
    uint4 *bc = reinterpret_cast<uint4 *>(tab + MOVE_TAB_BYTES); // [16] step pairs
    uint4 *trail = bc + 16;                                      // [16] what the walk left
    uint4 *ring = trail + 16;                                    // [MOVE_RING] proposals drawn ahead

    const int w = slot / s.m;
    const int lo = s.lo[w], hi = s.hi[w], nb = hi - lo + 1;
    const int kstart = s.k[slot];
    if (lo < 0 || nb < 1 || nb > s.W || kstart < lo || kstart > hi) { // malformed input: refuse
        if (lane == 0) atomicOr(&s.status->err, ERR_INPUT);
        return;
    }
    const double lnf = s.lnf[w];
    const bool frozen = s.finished[w] != 0;
    const int cfg = s.cfg ? s.cfg[slot] : slot;
    int8_t *gsp = s.spins + (size_t)cfg * s.spin_stride;
    const double *glng = s.lng + (size_t)slot * s.W;
    uint32_t *gH = s.H + (size_t)slot * s.W;
    const Lattice lat{s.L, s.N, s.magic};
    const int T = c.T;

    // ---- load lattice, shadow ln g
    if (s.vec_spins) {
        const int4 *src = reinterpret_cast<const int4 *>(gsp);
        uint4 *dst = reinterpret_cast<uint4 *>(cell);
        for (int i = lane; i < (s.N >> 4); i += 32) {
            const int4 v = src[i];
            dst[2 * i] = make_uint4(__byte_perm(v.x, ~0u, 0x4140), __byte_perm(v.x, ~0u, 0x4342),
                                    __byte_perm(v.y, ~0u, 0x4140), __byte_perm(v.y, ~0u, 0x4342));
            dst[2 * i + 1] = make_uint4(__byte_perm(v.z, ~0u, 0x4140), __byte_perm(v.z, ~0u, 0x4342),
                                        __byte_perm(v.w, ~0u, 0x4140), __byte_perm(v.w, ~0u, 0x4342));
        }
    } else {
        for (int i = lane; i < s.N; i += 32)
            cell[i] = (uint16_t)((NO_CLAIM << 8) | (uint8_t)gsp[i]);
    }
    double mx = 0.0;
    bool bad_in = false;
    for (int b = lane; b < nb; b += 32) {
        const double x = glng[b];
        bad_in = bad_in || !(fabs(x) < 0x1p30); // also catches NaN
        mx = fmax(mx, fabs(x));
        V[b] = bad_in ? 0LL : __double2ll_rn(__dmul_rn(x, 0x1p32));
    }
    // visited bits: the bins any walker of the window had visited when this launch started,
    // the start bin, and every bin this walker enters for the first time (always through the
    // float64 path below)
    // (replay has no window mask: every bin counts as visited there)
    const uint8_t *gmask = s.mask ? s.mask + (size_t)w * s.W : nullptr;
    for (int i = 0; i < visw(s.W); ++i) { // word i: bins 32i .. 32i+31, one per lane
        const int b = 32 * i + lane;
        const unsigned bits = __ballot_sync(FULL, b < nb && (gmask == nullptr || gmask[b]));
        if (lane == 0) vis[i] = bits;
    }
    __syncwarp();
    if (lane == 0) vis[(kstart - lo) >> 5] |= 1u << ((kstart - lo) & 31); // the start bin
    mx = warp_max(mx);
    // the shadow of a running window ends the launch below (max |ln g| + T ln f) 2^32 < 2^62,
    // and ln f 2^32 must not round to zero; a frozen window adds nothing to it
    const bool lnf_ok = frozen || (lnf >= 0x1p-32 && lnf < 0x1p20 && mx + (double)T * lnf < 0x1p30);
    if (__any_sync(FULL, bad_in) || !lnf_ok) {
        // the int64 shadow would overflow or lose the increment: leave the state untouched
        if (lane == 0) atomicOr(&s.status->err, ERR_RANGE);
        return;
    }
    const long long lnfq = __double2ll_rn(__dmul_rn(lnf, 0x1p32));
    const long long lnfq_add = frozen ? 0LL : lnfq;
    // interval-constant part of the float32 screening margin (ln units)
    const float Mbase = (float)(c.eps_l + 2.0 * shadow_error(mx, T, lnf, frozen) * 0x1p-32) * (1.0f + 0x1p-20f) + 0x1p-21f;
    const float lnf_f = frozen ? 0.0f : (float)lnf;
    const bool table_walk = lnf_f <= TABLE_WALK_LNF;
    // visits after which the ratio table is taken anew
    const int table_life = lnf_f > 0.0f ? (int)fminf(TABLE_DRIFT / lnf_f, 1e8f) : 100000000;

    const unsigned long long st0 = s.step[slot];
    unsigned int nacc = 0, nex = 0, nmis = 0; // nacc: of this lane's steps
    const uint32_t tag = (s.inst << 8) | TAG_MOVE;
    const unsigned below = (1u << lane) - 1u;
    // lane x counts the visits of cache bin x: bit i of x as a mask to xor a ballot with
    unsigned xinv[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) xinv[i] = ((lane >> i) & 1) ? 0u : ~0u;

    // The random words of step i.
    auto draw = [&](int i, uint32_t &w0, uint32_t &w1, uint32_t &w2) {
        if (REPLAY) {
            const uint32_t *wp = c.words + ((size_t)slot * T + i) * 3;
            w0 = i < T ? wp[0] : 0u;
            w1 = i < T ? wp[1] : 0u;
            w2 = i < T ? wp[2] : 0u;
        } else {
            const unsigned long long sn = st0 + (unsigned long long)i;
            const u32x4 r = philox((uint32_t)sn, (uint32_t)(sn >> 32), (uint32_t)(s.slot0 + slot), tag, s.key0,
                                   s.key1);
            w0 = r.x;
            w1 = r.y;
            w2 = r.z;
        }
    };
    // Proposals of steps g .. g+31 into the ring (when `room`): site and new-state draw, the four
    // neighbours, ln u.
    auto draw_ahead = [&](int g, bool room) {
        uint32_t w0, w1, w2;
        draw(g + lane, w0, w1, w2);
        const int site = (int)mulhi(w0, (uint32_t)s.N);
        int nl, nr, nu, nd;
        lat.nbrs(site, nl, nr, nu, nd);
        const unsigned pr = ISING ? 0u : mulhi(w1, (uint32_t)(s.q - 1));
        const uint4 e = make_uint4((unsigned)site | (pr << 16), (unsigned)nl | ((unsigned)nr << 16),
                                   (unsigned)nu | ((unsigned)nd << 16), __float_as_uint(lnu32(w2)));
        if (room) ring[(g + lane) & (MOVE_RING - 1)] = e;
    };

    // ---- the cached bins: lane j holds the shadow of bin wbase + j
    int wbase = kstart - 16, x = 16; // x: cache offset of the current bin
    bool bin_ok = false, far = false;
    long long Vr = 0;
    float Lw = 0.0f, M = 0.0f;
    auto cache_store = [&]() {
        if (bin_ok) V[wbase + lane - lo] = Vr;
        __syncwarp();
    };
    auto cache_load = [&](int k) {
        wbase = k - 16;
        x = 16;
        const int bj = wbase + lane;
        bin_ok = bj >= lo && bj <= hi;
        if (bin_ok) Vr = V[bj - lo];
        // Bins never visited keep their initial ln g while the others grow, so their cache
        // values can be far off: they are marked NaN (a step there is flagged unsure and
        // decided from the float64 values) and do not widen every other step's margin.
        far = bin_ok && !((vis[(bj - lo) >> 5] >> ((bj - lo) & 31)) & 1u);
    };
    // ln g of the cached bins relative to the current bin in float32, and the margin
    auto cache_floats = [&]() {
        const long long ref = __shfl_sync(FULL, Vr, x);
        const long long d = Vr - ref;
        Lw = __fmaf_rn(__uint2float_rn((uint32_t)d), 0x1p-32f, (float)(int)(d >> 32));
        // largest |Lw| of the cache (non-negative floats order like their bit patterns)
        const float Mx = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(bin_ok && !far ? fabsf(Lw) : 0.0f))) +
                         33.0f * lnf_f + 0x1p-20f;
        M = Mbase + 40.0f * ulpf(2.0f * Mx);
        if (!bin_ok) Lw = INFINITY; // a move there is rejected: ln g(k) - inf < ln u
        if (far) Lw = __int_as_float(0x7fc00000);
    };

    int g = 64; // steps drawn: always t + 2 NP at least
    draw_ahead(0, true);
    draw_ahead(32, true);
    cache_load(kstart);
    int table_age = table_life + 1; // visits since the table was taken
    __syncwarp();

    int t = 0;
    uint4 pe = ring[lane]; // lane j: the proposal of step t + j
    while (t < T) {
        const int n = min(2 * NP, T - t);
        const int site = (int)(pe.x & 0xffffu);
        if (lane < n) cellb[2 * site + 1] = (uint8_t)lane;
        __syncwarp();
        const unsigned c0 = cell[site], c1 = cell[pe.y & 0xffffu], c2 = cell[pe.y >> 16],
                       c3 = cell[pe.z & 0xffffu], c4 = cell[pe.z >> 16];
        const uint32_t nbytes = __byte_perm(__byte_perm(c1, c2, 0x0040), __byte_perm(c3, c4, 0x0040), 0x5410);
        const uint32_t s0 = c0 & 0xffu;
        // earlier lanes that propose one of this site's neighbours; settled after the walk: the
        // batch ends before the first step one of whose neighbours was changed
        unsigned claims = (shl_clamp(1u, c1 >> 8) | shl_clamp(1u, c2 >> 8) | shl_clamp(1u, c3 >> 8) |
                           shl_clamp(1u, c4 >> 8)) & below;
        bool dup = false; // an earlier lane proposes the same site: the batch ends before this step
        int snew, dkm;    // dkm = dk + DM
        if (ISING) {
            snew = -(int)(int8_t)s0;
            // dE = 2 s0 sum of neighbours, dk = dE / 4 = 2 - neighbours unequal to s0
            dkm = (int)__dp4a((int)bytes_unequal<true>(nbytes, s0), -1, 4);
        } else {
            snew = (int)(s0 + 1u + (pe.x >> 16));
            if (snew >= s.q) snew -= s.q;
            dkm = __dp4a((int)bytes_unequal<false>(nbytes, s0), -1,
                         __dp4a((int)bytes_unequal<false>(nbytes, (uint32_t)snew), 0x01010101, DM));
        }
        const int dk = dkm - DM;
        // a proposal that keeps the energy is always accepted and keeps the bin: the
        // walk sees it as a sure non-move (threshold +inf), the lane itself records the flip
        const bool dz = dk == 0;
        const float thr = dz ? INFINITY : __uint_as_float(pe.w);
        // two lanes on one site: make the lowest lane's claim stand
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
            claims = (shl_clamp(1u, cellb[2 * (pe.y & 0xffffu) + 1]) | shl_clamp(1u, cellb[2 * (pe.y >> 16) + 1]) |
                      shl_clamp(1u, cellb[2 * (pe.z & 0xffffu) + 1]) | shl_clamp(1u, cellb[2 * (pe.z >> 16) + 1])) & below;
        }
        __syncwarp();
        if (lane < n) cellb[2 * site + 1] = (uint8_t)NO_CLAIM;
        const bool cut = lane >= n || dup;

        // ---- the current bin near the edge of the cache: cache the bins around it
        if ((unsigned)(x - CACHE_LO) > (unsigned)(CACHE_HI - CACHE_LO)) {
            const int k = wbase + x;
            cache_store();
            cache_load(k);
            table_age = table_life + 1;
        }

        // ---- the walk: cache offsets xb, xa of the bin before and after step `lane`.  The batch
        // stops before step `stop`; `open` says that this step is not decided yet.
        int xb, xa, stop, scr = -1;
        bool open;
        auto stop_at = [&](bool accepted, bool ok) {
            const unsigned accs = __ballot_sync(FULL, accepted);
            const bool end = cut || (claims & accs) != 0u;
            const unsigned v = __reduce_min_sync(FULL, end ? 2u * lane : (ok ? 64u : 2u * lane + 1u));
            stop = (int)(v >> 1);
            open = v & 1u;
        };
        if (table_walk) {
            if (table_age > table_life) { // rows of the ratio table
                cache_floats();
#pragma unroll
                for (int d = 1; d <= DM; ++d) {
                    float up = __shfl_down_sync(FULL, Lw, d);
                    if (lane + d > 31) up = __int_as_float(0x7fc00000);
                    const __half h = __float2half_rn(Lw - up);
                    const int xd = (lane + d) & 31;
                    *reinterpret_cast<__half *>(tab + (DM + d) * ROW_BYTES + 4 * (lane & 15) + 2 * (lane >> 4)) = h;
                    *reinterpret_cast<__half *>(tab + (DM - d) * ROW_BYTES + 4 * (xd & 15) + 2 * (xd >> 4)) = __hneg(h);
                }
                table_age = 0;
                __syncwarp();
            }
            // the step is surely accepted from bin offset x if D(x) > tS, surely rejected if
            // D(x) < tR, whatever the visits since the table was taken did to ln g
            const float mg = __fmaf_rn((float)(table_age + lane + 1), lnf_f, M);
            const __half2 tS = __float2half2_rn(thr + mg);
            const __half tR = __float2half_rn(thr - mg);
            const unsigned char *row = tab + dkm * ROW_BYTES;
            unsigned S = 0u; // bit x: surely accepted from x
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const uint4 qv = reinterpret_cast<const uint4 *>(row)[v];
                const uint32_t ww[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    S |= __hgt2_mask(*reinterpret_cast<const __half2 *>(&ww[e]), tS) & (0x00010001u << (4 * v + e));
            }
            if (dz) S = 0u;
            const int dn = __shfl_down_sync(FULL, dk, 1);
            bool known = false; // step `lane` was decided below
            bool ok;
            // pairs of steps: from bin offset x the first one moves if bit x of a.x is set,
            // the second if bit x of a.y is set (whatever the first one did)
            auto publish = [&]() {
                const unsigned S1 = __shfl_down_sync(FULL, S, 1);
                const unsigned sh = __funnelshift_r(S1 << 4, S1 >> 28, (unsigned)(dk + 4)); // S1 seen from x + dk
                if (!(lane & 1)) bc[lane >> 1] = make_uint4(S, (S & sh) | (~S & S1), (unsigned)dk, (unsigned)dn);
                __syncwarp();
            };
            auto walk = [&]() {
                int y = 31 - x; // S << y has the bit of offset x on top
                unsigned pk[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const uint4 a = bc[p];
                    pk[p >> 2] |= (unsigned)y << (8 * (p & 3));
                    const int m0 = sign_mask((int)(a.x << y)), m1 = sign_mask((int)(a.y << y));
                    y += m0 * (int)a.z;
                    y += m1 * (int)a.w;
                }
                const uint4 a = bc[lane >> 1];
                const unsigned pw = lane < 16 ? (lane < 8 ? pk[0] : pk[1]) : (lane < 24 ? pk[2] : pk[3]);
                const int yq = (int)((pw >> (8 * ((lane >> 1) & 3))) & 31u);
                const int m0 = sign_mask((int)(a.x << yq)), m1 = sign_mask((int)(a.y << yq));
                const int odd = -(lane & 1);
                xb = 31 - yq + (m0 & odd & (int)a.z);
                const int mv = pick(odd, m1, m0);
                xa = xb + (mv & dk);
                const __half D = *reinterpret_cast<const __half *>(row + 4 * (xb & 15) + 2 * ((xb >> 4) & 1));
                ok = dz || mv != 0 || known || __hlt(D, tR);
                if (CHECK) ok = dz || (unsigned)(xb + dk - (lo - wbase)) >= (unsigned)nb;
                stop_at(dz || mv != 0, ok);
            };
            publish();
            if (NP == 16) { // the walk leaves most issue slots idle: draw proposals in them
                const bool room = g + 32 - t <= MOVE_RING;
                draw_ahead(g, room);
                g += room ? 32 : 0;
            }
            walk();
            while (open) {
                // step `stop`: its ln g difference with the visits before it, in float32
                const int u = stop;
                const int xu = __shfl_sync(FULL, xb, u), du = __shfl_sync(FULL, dk, u);
                const int xt = xu + du;
                if ((unsigned)xt >= 32u) {
                    open = u == 0; // else the next batch's cache will hold the target
                    break;
                }
                if (table_age > 0) { // bring the cached values up to date
                    const float Mt = M;
                    cache_floats();
                    M = fmaxf(M, Mt);
                }
                const unsigned bu = (1u << u) - 1u;
                const int cx = __popc(__ballot_sync(FULL, xa == xu) & bu), ct = __popc(__ballot_sync(FULL, xa == xt) & bu);
                const float e = __fmaf_rn((float)(cx - ct), lnf_f, __shfl_sync(FULL, Lw, xu) - __shfl_sync(FULL, Lw, xt)) -
                                __shfl_sync(FULL, thr, u);
                if (CHECK) {
                    const int sure = ((S >> xu) & 1u) ? 1 : (__hlt(*reinterpret_cast<const __half *>(
                                                                 row + 4 * (xu & 15) + 2 * (xu >> 4)), tR) ? 0 : -1);
                    scr = __shfl_sync(FULL, sure, u);
                    if (scr < 0) scr = e > M ? 1 : (e < -M ? 0 : -1);
                    break;
                }
                if (!(fabsf(e) > M)) break; // too close: float64
                if (lane == u) {
                    known = true;
                    if (e > M) S |= 1u << xu;
                }
                publish();
                walk();
            }
            table_age += stop;
        } else {
            // Large ln f: the visits of the batch decide its later steps, so the path is walked
            // with running float32 values.  Steps are resolved in pairs: the three cache
            // lookups a pair can need (k' of the first step; k' of the second after the first
            // moved / stayed) are issued together and the second step is evaluated in both
            // worlds, so one shuffle latency covers two moves.  Decision variable:
            // v = M - (ln g(k) - ln g(k') - thr); accept if v < 0, reject if v > 2M, else unsure.
            // Outcomes are sign masks, not predicates: a predicate takes more than twice the
            // cycles of an integer operation before it can be used.
            // A target outside the 32 cached bins reads a wrong lane; such steps are found after
            // the loop and cut there as well.
            cache_floats();
            reinterpret_cast<uint2 *>(bc)[lane] = make_uint2(__float_as_uint(thr + M), (unsigned)dk);
            if (NP == 16) {
                const bool room = g + 32 - t <= MOVE_RING;
                draw_ahead(g, room);
                g += room ? 32 : 0;
            }
            __syncwarp();
            float Lr = Lw;   // the cache, with the running values of the bins left
            int xk = x;      // cache offset of the current bin
            float Lk = 0.0f; // its running value (the cache holds it only once left)
#pragma unroll 4
            for (int p = 0; p < NP; ++p) {
                const uint4 a = bc[p];
                const int d0 = (int)a.y, d1 = (int)a.w;
                const int x0 = xk + d0; // k' of step i
                const int xA = x0 + d1; // k' of step i+1 if step i moved
                const int xR = xk + d1; // k' of step i+1 if step i stayed
                const float L0 = __shfl_sync(FULL, Lr, x0);
                const float LA_ = __shfl_sync(FULL, Lr, xA);
                const float LR = __shfl_sync(FULL, Lr, xR);
                const float LA = (d1 == -d0) ? Lk : LA_; // back to the bin just left
                const int onk = lane == xk ? -1 : 0, on0 = lane == x0 ? -1 : 0;
                const float Ls = Lk + lnf_f; // value after step i if stayed
                const float Lm = L0 + lnf_f; // value after step i if moved
                const float v0 = (__uint_as_float(a.x) - Lk) + L0;
                const int m0 = sign_mask(__float_as_int(v0));
                const float v1 = pickf(m0, (__uint_as_float(a.z) - Lm) + LA, (__uint_as_float(a.z) - Ls) + LR);
                const int m1 = sign_mask(__float_as_int(v1));
                const int xc = pick(m0, x0, xk);
                const float Lc = pickf(m0, Lm, Ls);
                Lr = pickf(m0 & onk, Lk, Lr); // the bins left keep their running values
                Lr = pickf(m1 & pick(m0, on0, onk), Lc, Lr);
                xk = pick(m1, pick(m0, xA, xR), xc);
                Lk = pickf(m1, pickf(m0, LA, LR), Lc) + lnf_f;
                if (lane == 0) // one lane: a store by all of them holds the shuffles up behind it
                    trail[p] = make_uint4((unsigned)xc, __float_as_uint(v0), (unsigned)xk, __float_as_uint(v1));
            }
            __syncwarp();
            const uint2 tr = reinterpret_cast<const uint2 *>(trail)[lane];
            xa = (int)tr.x;
            const float v = __uint_as_float(tr.y);
            const int xup = __shfl_up_sync(FULL, xa, 1);
            xb = lane == 0 ? x : xup;
            const bool oob = (unsigned)(xb + dk) >= 32u;
            bool ok = (v < 0.0f || v > 2.0f * M * (1.0f + 0x1p-20f)) && !oob;
            if (CHECK) ok = dz || (unsigned)(xb + dk - (lo - wbase)) >= (unsigned)nb;
            stop_at(dz || xa != xb, ok);
            if (open) {
                const bool out = __shfl_sync(FULL, oob ? 1 : 0, stop);
                if (CHECK) {
                    const float vu = __shfl_sync(FULL, v, stop);
                    scr = out ? -1 : (vu < 0.0f ? 1 : (vu > 2.0f * M * (1.0f + 0x1p-20f) ? 0 : -1));
                } else if (stop > 0 && out) {
                    open = false; // the next batch's cache will hold the target
                    table_age = table_life + 1;
                }
            }
        }
        if (stop == 0 && !open) { // no step done and none to decide: cannot happen (lane 0 is never cut)
            if (lane == 0) atomicOr(&s.status->err, ERR_INPUT);
            return;
        }

        // ---- side effects of steps 0 .. stop-1
        const bool mine = lane < stop;
        const bool accj = dz || xa != xb; // step j accepted (a move to another bin, or dE = 0)
        if (mine && accj) cellb[2 * site] = (uint8_t)snew; // distinct sites
        t += stop;
        const uint4 pnext = ring[(t + lane) & (MOVE_RING - 1)];
        const int step_done = t - stop;
        {
            // visits: lane x counts the steps that ended in cache bin x
            unsigned v = stop < 32 ? (1u << stop) - 1u : FULL;
#pragma unroll
            for (int i = 0; i < 5; ++i) v &= __ballot_sync(FULL, (xa >> i) & 1) ^ xinv[i];
            Vr += (long long)__popc(v) * lnfq_add;
        }
        if (REPLAY && mine) {
            c.acc_out[(size_t)slot * T + step_done + lane] = accj ? 1 : 0;
            c.dk_out[(size_t)slot * T + step_done + lane] = dk;
        }
        nacc += mine && accj ? 1u : 0u;
        if (stop > 0) x = __shfl_sync(FULL, xa, stop - 1);
        pe = pnext;
        __syncwarp();

        // ---- a proposal too close to call in float32: decide it from the float64 values
        if (open) {
            const int dki = __shfl_sync(FULL, dk, stop);
            const int sitei = __shfl_sync(FULL, site, stop);
            const int snewi = __shfl_sync(FULL, snew, stop);
            int k = wbase + x;
            const int kp = k + dki;
            bool acc = dki == 0;
            cache_store();
            if (!acc && kp >= lo && kp <= hi) {
                uint32_t w0, w1, w2i;
                draw(t, w0, w1, w2i);
                acc = exact_decision(glng, V, lo, k, kp, lnf, lnfq, frozen, w2i);
                if (scr < 0) ++nex;
                else if ((int)acc != scr) ++nmis;
            }
            __syncwarp();
            if (acc) {
                k = kp;
                if (lane == 0) {
                    cellb[2 * sitei] = (uint8_t)snewi;
                    ++nacc;
                }
            }
            if (lane == 0) {
                V[k - lo] += lnfq_add;
                // a bin reached for the first time is only ever entered here (its cache value
                // is NaN until marked), so marking it here keeps the visited set complete
                vis[(k - lo) >> 5] |= 1u << ((k - lo) & 31);
            }
            if (REPLAY && lane == 0) {
                c.acc_out[(size_t)slot * T + t] = acc ? 1 : 0;
                c.dk_out[(size_t)slot * T + t] = dki;
            }
            t += 1;
            pe = ring[(t + lane) & (MOVE_RING - 1)];
            __syncwarp();
            cache_load(k);
            table_age = table_life + 1;
        }
        if (NP < 16 && g < t + 64) { // several small batches use up one draw of 32
            draw_ahead(g, true);
            g += 32;
            __syncwarp();
        }
    }
    cache_store();

    // ---- write back lattice, float64 ln g (rebuilt exactly), H, counters
    if (s.vec_spins) {
        const uint4 *src = reinterpret_cast<const uint4 *>(cell);
        int4 *dst = reinterpret_cast<int4 *>(gsp);
        for (int i = lane; i < (s.N >> 4); i += 32) {
            const uint4 a = src[2 * i], b = src[2 * i + 1];
            dst[i] = make_int4(__byte_perm(a.x, a.y, 0x6420), __byte_perm(a.z, a.w, 0x6420),
                               __byte_perm(b.x, b.y, 0x6420), __byte_perm(b.z, b.w, 0x6420));
        }
    } else {
        for (int i = lane; i < s.N; i += 32) gsp[i] = (int8_t)(cell[i] & 0xffu);
    }
    if (!frozen) {
        double *gl = s.lng + (size_t)slot * s.W;
        for (int b = lane; b < nb; b += 32) {
            const uint32_t v = visits(V, gl, b, lnfq);
            if (v != 0u) {
                gl[b] = seqadd(gl[b], lnf, v);
                gH[b] += v;
            }
        }
    }
    nacc = __reduce_add_sync(FULL, nacc);
    if (lane == 0) {
        s.k[slot] = wbase + x;
        s.step[slot] = st0 + (unsigned long long)T;
        s.acc[slot] += nacc;
        if (nex) atomicAdd(&s.status->n_exact, (unsigned long long)nex);
        if (nmis) atomicAdd(&s.status->n_mismatch, (unsigned long long)nmis);
    }
}

template <bool ISING, bool REPLAY, bool CHECK>
__device__ __forceinline__ void move_walker(const State &s, const MoveCfg &c, const int slot,
                                            unsigned char *base, const int lane)
{
    if (s.status != nullptr && s.status->done) return;
    if (s.N >= BATCH32_SITES) move_walker_n<ISING, REPLAY, CHECK, 16>(s, c, slot, base, lane);
    else if (s.N >= BATCH16_SITES) move_walker_n<ISING, REPLAY, CHECK, 8>(s, c, slot, base, lane);
    else move_walker_n<ISING, REPLAY, CHECK, 4>(s, c, slot, base, lane);
}

// ---------------------------------------------------------------------------------------
// One thread per walker (small lattices, many walkers): the plain sequential walk of Sec. 2.
// ln g is the same int64 shadow as above (multiples of 2^-32, exact visit counts), held in
// shared memory; the current bin's value stays in registers.  Each decision is screened in
// fixed point: D = V(k) - V(k') against ln u 2^32 (the float32 value, converted exactly up to
// one unit), accepted or rejected when |D - ln u 2^32| exceeds the margin Mq that bounds the
// shadow error, the float32 ln u error and the float64 rounding of ln g(k) - ln g(k'); inside
// the margin the float64 values are rebuilt (rare).  No float arithmetic in the loop, no
// warp cooperation: the 32 walkers of a warp run in lockstep, each on its own data.
// ---------------------------------------------------------------------------------------
template <bool ISING, bool REPLAY, bool CHECK>
__device__ __forceinline__ void move_walker_thread(const State &s, const MoveCfg &c, const int slot,
                                                   unsigned char *base)
{
    if (s.status != nullptr && s.status->done) return;
    int8_t *sp = reinterpret_cast<int8_t *>(base);
    long long *V = reinterpret_cast<long long *>(base + pad16(s.N));
    const int w = slot / s.m;
    const int lo = s.lo[w], hi = s.hi[w], nb = hi - lo + 1;
    int k = s.k[slot];
    if (lo < 0 || nb < 1 || nb > s.W || k < lo || k > hi) {
        atomicOr(&s.status->err, ERR_INPUT);
        return;
    }
    const double lnf = s.lnf[w];
    const bool frozen = s.finished[w] != 0;
    const int cfg = s.cfg ? s.cfg[slot] : slot;
    int8_t *gsp = s.spins + (size_t)cfg * s.spin_stride;
    double *glng = s.lng + (size_t)slot * s.W;
    uint32_t *gH = s.H + (size_t)slot * s.W;
    const Lattice lat{s.L, s.N, s.magic};
    const int T = c.T;
    if (s.vec_spins) {
        const int4 *src = reinterpret_cast<const int4 *>(gsp);
        int4 *dst = reinterpret_cast<int4 *>(sp);
        for (int i = 0; i < (s.N >> 4); ++i) dst[i] = src[i];
    } else {
        for (int i = 0; i < s.N; ++i) sp[i] = gsp[i];
    }
    double mx = 0.0;
    bool bad = false;
    for (int b = 0; b < nb; ++b) {
        const double x = glng[b];
        bad = bad || !(fabs(x) < 0x1p30);
        mx = fmax(mx, fabs(x));
        V[b] = bad ? 0LL : __double2ll_rn(__dmul_rn(x, 0x1p32));
    }
    const bool lnf_ok = frozen || (lnf >= 0x1p-32 && lnf < 0x1p20 && mx + (double)T * lnf < 0x1p30);
    if (bad || !lnf_ok) {
        atomicOr(&s.status->err, ERR_RANGE);
        return;
    }
    const long long lnfq = frozen ? 0LL : __double2ll_rn(__dmul_rn(lnf, 0x1p32));
    // margin in units of 2^-32: both shadow values, the float32 ln u, the float64 difference
    // of ln g values below 2^31 (half an ulp, 2^-22) and the conversion of ln u (one unit)
    const long long Mq = (long long)(2.0 * shadow_error(mx, T, lnf, frozen) + (c.eps_l + 0x1p-21) * 0x1p32) + 4;
    const unsigned long long st0 = s.step[slot];
    const uint32_t tag = (s.inst << 8) | TAG_MOVE;
    unsigned int nacc = 0, nex = 0, nmis = 0;
    long long Vk = V[k - lo];
    for (int t = 0; t < T; ++t) {
        uint32_t w0, w1, w2;
        if (REPLAY) {
            const uint32_t *wp = c.words + ((size_t)slot * T + t) * 3;
            w0 = wp[0];
            w1 = wp[1];
            w2 = wp[2];
        } else {
            const unsigned long long sn = st0 + (unsigned long long)t;
            const u32x4 r = philox((uint32_t)sn, (uint32_t)(sn >> 32), (uint32_t)(s.slot0 + slot),
                                   tag, s.key0, s.key1);
            w0 = r.x;
            w1 = r.y;
            w2 = r.z;
        }
        const int site = (int)mulhi(w0, (uint32_t)s.N);
        const int pr = ISING ? 0 : (int)mulhi(w1, (uint32_t)(s.q - 1));
        int snew;
        const int dk = propose_dk<ISING>(sp, lat, s.q, site, pr, snew);
        const int kp = k + dk;
        bool acc = dk == 0;
        if (!acc && kp >= lo && kp <= hi) {
            const long long e = (Vk - V[kp - lo]) - (long long)__float2ll_rz(lnu32(w2) * 0x1p32f);
            const int scr = e > Mq ? 1 : (e < -Mq ? 0 : -1);
            if (scr >= 0 && !CHECK) {
                acc = scr == 1;
            } else {
                V[k - lo] = Vk;
                acc = exact_value_decision(glng, V, lo, k, kp, lnf, lnfq, frozen, w2);
                if (scr < 0) ++nex;
                else if ((int)acc != scr) ++nmis;
            }
        }
        if (acc) {
            sp[site] = (int8_t)snew;
            if (dk != 0) {
                V[k - lo] = Vk;
                k = kp;
                Vk = V[k - lo];
            }
            ++nacc;
        }
        Vk += lnfq; // ln g(k) += ln f, H(k)++: one visit of the current bin
        if (REPLAY) {
            c.acc_out[(size_t)slot * T + t] = acc ? 1 : 0;
            c.dk_out[(size_t)slot * T + t] = dk;
        }
    }
    V[k - lo] = Vk;
    if (s.vec_spins) {
        const int4 *src = reinterpret_cast<const int4 *>(sp);
        int4 *dst = reinterpret_cast<int4 *>(gsp);
        for (int i = 0; i < (s.N >> 4); ++i) dst[i] = src[i];
    } else {
        for (int i = 0; i < s.N; ++i) gsp[i] = sp[i];
    }
    if (!frozen)
        for (int b = 0; b < nb; ++b) {
            const uint32_t v = visits(V, glng, b, lnfq);
            if (v != 0u) {
                glng[b] = seqadd(glng[b], lnf, v);
                gH[b] += v;
            }
        }
    s.k[slot] = k;
    s.step[slot] = st0 + (unsigned long long)T;
    s.acc[slot] += nacc;
    if (nex) atomicAdd(&s.status->n_exact, (unsigned long long)nex);
    if (nmis) atomicAdd(&s.status->n_mismatch, (unsigned long long)nmis);
}

template <bool ISING, bool REPLAY, bool CHECK>
__global__ void __launch_bounds__(256) k_move_thread(State s, MoveCfg c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int slot = blockIdx.x * c.walkers_per_block + threadIdx.x;
    if (threadIdx.x >= c.walkers_per_block || slot >= s.nw) return;
    move_walker_thread<ISING, REPLAY, CHECK>(s, c, slot,
                                             smem + (size_t)threadIdx.x * move_smem_per_thread_walker(s.N, s.W));
}

template <bool ISING, bool REPLAY, bool CHECK>
__global__ void __launch_bounds__(512, 1) k_move(State s, MoveCfg c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int slot = blockIdx.x * c.walkers_per_block + wib;
    if (slot >= s.nw) return;
    move_walker<ISING, REPLAY, CHECK>(s, c, slot, smem + (size_t)wib * move_smem_per_walker(s.N, s.W),
                                      lane);
}

// Batched instances in one launch: CTA b serves walkers jobs[b].y .. jobs[b].y + jobs[b].z - 1 of
// instance jobs[b].x & 0xffffff, one warp per walker, or one thread per walker when bit 24 of
// jobs[b].x is set; the model and the layout are chosen per CTA.
template <bool CHECK>
__global__ void __launch_bounds__(512, 1) k_move_batch(const State *__restrict__ states,
                                                    const int4 *__restrict__ jobs, MoveCfg c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int4 job = jobs[blockIdx.x];
    const State s = states[job.x & 0xffffff];
    if (job.x >> 24) { // one thread per walker
        const int t = threadIdx.x;
        if (t >= job.z) return;
        unsigned char *base = smem + (size_t)t * move_smem_per_thread_walker(s.N, s.W);
        if (s.model == 0) move_walker_thread<true, false, CHECK>(s, c, job.y + t, base);
        else move_walker_thread<false, false, CHECK>(s, c, job.y + t, base);
        return;
    }
    if (wib >= job.z) return;
    unsigned char *base = smem + (size_t)wib * move_smem_per_walker(s.N, s.W);
    if (s.model == 0) move_walker<true, false, CHECK>(s, c, job.y + wib, base, lane);
    else move_walker<false, false, CHECK>(s, c, job.y + wib, base, lane);
}

cudaError_t launch_move_batch(const State *states, const int4 *jobs, int njobs, int walkers_per_block,
                              size_t smem, const MoveCfg &c, cudaStream_t st)
{
    if (njobs <= 0) return cudaSuccess;
    cudaError_t e;
    if (c.check_all) {
        e = cudaFuncSetAttribute(k_move_batch<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_move_batch<true><<<njobs, 32 * walkers_per_block, smem, st>>>(states, jobs, c);
    } else {
        e = cudaFuncSetAttribute(k_move_batch<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_move_batch<false><<<njobs, 32 * walkers_per_block, smem, st>>>(states, jobs, c);
    }
    return cudaGetLastError();
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
    const dim3 grid((s.nw + G - 1) / G), block(32 * G);
    const bool ising = s.model == 0;
    cudaError_t e;
#define REWL_LAUNCH_MOVE(I, R, C)                                                                \
    do {                                                                                         \
        e = cudaFuncSetAttribute(k_move<I, R, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                                 (int)smem);                                                     \
        if (e != cudaSuccess) return e;                                                          \
        k_move<I, R, C><<<grid, block, smem, st>>>(s, c);                                        \
    } while (0)
    if (ising) {
        if (c.words) REWL_LAUNCH_MOVE(true, true, false);
        else if (c.check_all) REWL_LAUNCH_MOVE(true, false, true);
        else REWL_LAUNCH_MOVE(true, false, false);
    } else {
        if (c.words) REWL_LAUNCH_MOVE(false, true, false);
        else if (c.check_all) REWL_LAUNCH_MOVE(false, false, true);
        else REWL_LAUNCH_MOVE(false, false, false);
    }
#undef REWL_LAUNCH_MOVE
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Seeded lattices and prep into the window: one warp per walker, the lattice in shared memory
// (cells as in the move kernel).  Far from the window a proposal is accepted by the sign of its
// energy change alone, so a batch of 32 has no serial part but its conflicts (a site proposed
// twice, or a neighbour that an earlier step of the batch changed: the batch ends there); near it
// a prefix sum finds the step that reaches the window, and that step is decided by itself.
// Bound by the latency of a batch.  Potts q=10 L=80, 1024 walkers, rewl_init with the lattices
// and bins read back: 548 ms with one thread per walker on global memory, 7.7 ms with a warp each.
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
        while (dist_to(k, lo, hi) > 0 && ps < end) {
            const int n = (int)min(32ULL, end - ps);
            const unsigned long long i = ps + (unsigned long long)lane;
            const u32x4 r = philox((uint32_t)i, (uint32_t)(i >> 32), (uint32_t)(s.slot0 + slot),
                                   (s.inst << 8) | TAG_PREP, s.key0, s.key1);
            const int site = (int)mulhi(r.x, (uint32_t)N);
            int nl, nr, nu, nd;
            lat.nbrs(site, nl, nr, nu, nd);
            // claims: the lowest lane that proposes a site marks it
            if (lane < n) cellb[2 * site + 1] = (uint8_t)lane;
            __syncwarp();
            unsigned own = cellb[2 * site + 1];
            for (int it = 0; it < 32; ++it) { // each pass lowers some claim: ends within 32 passes
                const bool again = lane < n && own > (unsigned)lane;
                if (!__any_sync(FULL, again)) break;
                if (again) cellb[2 * site + 1] = (uint8_t)lane;
                __syncwarp();
                own = cellb[2 * site + 1];
                __syncwarp();
            }
            const bool dup = lane < n && own < (unsigned)lane;
            const unsigned c1 = cell[nl], c2 = cell[nr], c3 = cell[nu], c4 = cell[nd];
            const uint32_t s0 = cell[site] & 0xffu;
            const unsigned claims = (shl_clamp(1u, c1 >> 8) | shl_clamp(1u, c2 >> 8) | shl_clamp(1u, c3 >> 8) |
                                     shl_clamp(1u, c4 >> 8)) & below;
            const uint32_t nbytes = __byte_perm(__byte_perm(c1, c2, 0x0040), __byte_perm(c3, c4, 0x0040), 0x5410);
            int snew, dk;
            if (ISING) {
                snew = -(int)(int8_t)s0;
                dk = 2 - __popc(bytes_unequal<true>(nbytes, s0));
            } else {
                snew = (int)s0 + 1 + (int)mulhi(r.y, (uint32_t)(s.q - 1));
                if (snew >= s.q) snew -= s.q;
                dk = __popc(bytes_unequal<false>(nbytes, (uint32_t)snew)) - __popc(bytes_unequal<false>(nbytes, s0));
            }
            __syncwarp();
            if (lane < n) cellb[2 * site + 1] = (uint8_t)NO_CLAIM;
            // accepted while the walker stays on its side of the window
            const bool above = k > hi;
            bool acc = above ? dk <= 0 : dk >= 0;
            const unsigned accs = __ballot_sync(FULL, acc);
            int done = (int)__reduce_min_sync(FULL, lane >= n || dup || (claims & accs) ? (unsigned)lane : 32u);
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
// Flatness + window advance (Sec. 2).  One CTA per window.
// ---------------------------------------------------------------------------------------
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
#pragma unroll 4
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

__global__ void k_check(State s, double flatness, double lnf_final)
{
    check_window(s, blockIdx.x, flatness, lnf_final);
}

// tab[b] = (instance, window); prm[instance] = (flatness, ln f_final)
__global__ void k_check_batch(const State *__restrict__ states, const int2 *__restrict__ tab,
                              const double2 *__restrict__ prm)
{
    const int2 t = tab[blockIdx.x];
    const State s = states[t.x];
    const double2 p = prm[t.x];
    check_window(s, t.y, p.x, p.y);
}

cudaError_t launch_check_batch(const State *states, const int2 *tab, int n, const double2 *prm,
                               cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_check_batch<<<n, 512, 0, st>>>(states, tab, prm);
    return cudaGetLastError();
}

cudaError_t launch_check(const State &s, double flatness, double lnf_final, cudaStream_t st)
{
    k_check<<<s.h, 512, 0, st>>>(s, flatness, lnf_final);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Replica exchange (Eq. 1) between windows (w, w+1), w = round mod 2.  One warp per pair;
// lane 0 draws the partner permutation and the decisions (m is small), the swap itself
// exchanges configuration indices and bins.
// ---------------------------------------------------------------------------------------
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

__device__ __forceinline__ void swap_pair(const State &s, const int pair)
{
    // one warp per window pair: the permutation's random draws and the m exchange decisions
    // are lane-parallel (each decision touches its own two walker slots); only the
    // Fisher-Yates swaps themselves run in order.  Pairs (w, w+1) with the global window
    // index w0 + w of the parity of the round.
    if (s.status->done) return;
    const long long rd = s.status->round;
    const int w = 2 * pair + (int)((rd + s.w0) & 1);
    if (w + 1 >= s.h) return;
    const int lane = threadIdx.x & 31;
    const int m = s.m, W = s.W;
    __shared__ int perm[MAX_M];
    __shared__ int draw[MAX_M];
    exchange_perm(s, s.w0 + w, rd, perm, draw);
    const int loA = s.lo[w], hiA = s.hi[w], loB = s.lo[w + 1], hiB = s.hi[w + 1];
    unsigned acc = 0;
    for (int i = lane; i < m; i += 32) {
        const int a = w * m + i, b = (w + 1) * m + perm[i];
        const int kx = s.k[a], ky = s.k[b];
        if (kx < loB || kx > hiB || ky < loA || ky > hiA) continue;
        const double *ga = s.lng + (size_t)a * W, *gb = s.lng + (size_t)b * W;
        const double lnP = __dadd_rn(__dsub_rn(ga[kx - loA], ga[ky - loA]),
                                     __dsub_rn(gb[ky - loB], gb[kx - loB]));
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

__global__ void k_swap(State s) { swap_pair(s, blockIdx.x); }

// tab[b] = (instance, pair index)
__global__ void k_swap_batch(const State *__restrict__ states, const int2 *__restrict__ tab)
{
    const int2 t = tab[blockIdx.x];
    const State s = states[t.x];
    swap_pair(s, t.y);
}

cudaError_t launch_swap_batch(const State *states, const int2 *tab, int n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_swap_batch<<<n, 32, 0, st>>>(states, tab);
    return cudaGetLastError();
}

cudaError_t launch_swap(const State &s, cudaStream_t st)
{
    if (s.h < 2) return cudaSuccess;
    k_swap<<<(s.h + 1) / 2, 32, 0, st>>>(s);
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

__device__ __forceinline__ void round_end(const State &s)
{
    if (s.status->done) return;
    s.status->round += 1;
    int all = !s.production;
    for (int w = 0; w < s.h; ++w) all &= s.finished[w];
    if (all) s.status->done = 1;
}

__global__ void k_round_end(State s) { round_end(s); }

__global__ void k_round_end_batch(const State *__restrict__ states, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) round_end(states[i]);
}

cudaError_t launch_round_end_batch(const State *states, int n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_round_end_batch<<<(n + 63) / 64, 64, 0, st>>>(states, n);
    return cudaGetLastError();
}

cudaError_t launch_round_end(const State &s, cudaStream_t st)
{
    k_round_end<<<1, 1, 0, st>>>(s);
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

// One CTA: joins are found pair by pair (each depends on the previous one); the stencils
// and the argmin over the overlap are block-parallel.
__global__ void k_stitch(State s, const double *mean, double de, int step, int norm, double target,
                         double *out, int *joins, int *ok, int B)
{
    const int W = s.W;
    __shared__ double shift_s;
    __shared__ int prev_s, fail_s;
    for (int b = threadIdx.x; b <= B; b += blockDim.x) out[b] = -INFINITY;
    __syncthreads();
    {
        const int lo0 = s.lo[0], hi0 = s.hi[0];
        for (int b = lo0 + (int)threadIdx.x; b <= hi0; b += blockDim.x)
            if (s.mask[b - lo0]) out[b] = mean[b - lo0];
    }
    if (threadIdx.x == 0) {
        shift_s = 0.0;
        prev_s = -1;
        fail_s = 0;
    }
    __syncthreads();
    for (int w = 0; w + 1 < s.h; ++w) {
        const double *la = mean + (size_t)w * W, *lb = mean + (size_t)(w + 1) * W;
        const uint8_t *va = s.mask + (size_t)w * W, *vb = s.mask + (size_t)(w + 1) * W;
        const int loa = s.lo[w], hia = s.hi[w], lob = s.lo[w + 1], hib = s.hi[w + 1];
        const int nba = hia - loa + 1, nbb = hib - lob + 1;
        const int prev = prev_s;
        int kj = -1;
        for (int npts = 5; npts >= 3 && kj < 0; npts -= 2) {
            double best = INFINITY;
            int bk = 0x7fffffff;
            for (int k = lob + (int)threadIdx.x; k <= hia; k += blockDim.x) {
                if (k <= prev || !va[k - loa] || !vb[k - lob]) continue;
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
            if (best < INFINITY) kj = bk;
        }
        if (kj < 0) { // nearest bin valid in both to the overlap midpoint, ties -> smaller
            const int mid2 = lob + hia;
            double bd = INFINITY;
            int bk = 0x7fffffff;
            for (int k = lob + (int)threadIdx.x; k <= hia; k += blockDim.x) {
                if (k <= prev || !va[k - loa] || !vb[k - lob]) continue;
                const double d = fabs((double)(2 * k - mid2));
                if (d < bd || (d == bd && k < bk)) {
                    bd = d;
                    bk = k;
                }
            }
            block_argmin(bd, bk);
            if (bd < INFINITY) kj = bk;
        }
        if (kj < 0) {
            if (threadIdx.x == 0) fail_s = 1;
            break;
        }
        if (threadIdx.x == 0) {
            shift_s = __dsub_rn(__dadd_rn(la[kj - loa], shift_s), lb[kj - lob]);
            joins[w] = kj;
            prev_s = kj;
        }
        __syncthreads();
        const double sh = shift_s;
        for (int b = max(kj, lob) + (int)threadIdx.x; b <= hib; b += blockDim.x)
            out[b] = vb[b - lob] ? __dadd_rn(lb[b - lob], sh) : -INFINITY;
        __syncthreads();
    }
    __syncthreads();
    if (fail_s) {
        if (threadIdx.x == 0) *ok = 0;
        return;
    }
    if (norm == 0) {
        double mx = -INFINITY;
        for (int b = threadIdx.x; b <= B; b += blockDim.x) mx = fmax(mx, out[b]);
        mx = block_reduce_max(mx);
        double sum = 0.0;
        for (int b = threadIdx.x; b <= B; b += blockDim.x)
            if (out[b] > -INFINITY) sum += exp(out[b] - mx);
        sum = block_reduce_sum(sum);
        const double cst = (mx + log(sum)) - target;
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

cudaError_t launch_stitch(const State &s, const double *mean, double de, int step, int norm,
                          double target, double *out, int *joins, int *ok, int B, cudaStream_t st)
{
    k_stitch<<<1, 256, 0, st>>>(s, mean, de, step, norm, target, out, joins, ok, B);
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

// ---------------------------------------------------------------------------------------
// Canonical averages from ln g (Eqs. 6-7): one CTA per temperature; u = <E>/N,
// c = <(E - <E>)^2> / (N T^2), weights g(E) e^{-E/T} taken relative to their maximum.
// ---------------------------------------------------------------------------------------
__global__ void k_thermo(const double *__restrict__ lng, int B, int model, int N,
                         const double *__restrict__ Ts, double *__restrict__ U,
                         double *__restrict__ Cv)
{
    const double T = Ts[blockIdx.x];
    auto energy = [&](int b) { return -2.0 * N + (model == 0 ? 4.0 * b : (double)b); };
    double mx = -INFINITY;
    for (int b = threadIdx.x; b <= B; b += blockDim.x)
        if (lng[b] > -INFINITY) mx = fmax(mx, lng[b] - energy(b) / T);
    mx = block_reduce_max(mx);
    double s0 = 0.0, s1 = 0.0;
    for (int b = threadIdx.x; b <= B; b += blockDim.x)
        if (lng[b] > -INFINITY) {
            const double w = exp(lng[b] - energy(b) / T - mx);
            s0 += w;
            s1 += w * energy(b);
        }
    s0 = block_reduce_sum(s0);
    s1 = block_reduce_sum(s1);
    const double e1 = s1 / s0;
    double s2 = 0.0;
    for (int b = threadIdx.x; b <= B; b += blockDim.x)
        if (lng[b] > -INFINITY) {
            const double w = exp(lng[b] - energy(b) / T - mx);
            const double de = energy(b) - e1;
            s2 += w * de * de;
        }
    s2 = block_reduce_sum(s2);
    if (threadIdx.x == 0) {
        U[blockIdx.x] = e1 / N;
        Cv[blockIdx.x] = s2 / s0 / ((double)N * T * T);
    }
}

cudaError_t launch_thermo(const double *lng, int model, int L, const double *T, int nT, double *U,
                          double *C, cudaStream_t st)
{
    if (nT <= 0) return cudaSuccess;
    const int N = L * L, B = model == 0 ? N : 2 * N;
    k_thermo<<<nT, 256, 0, st>>>(lng, B, model, N, T, U, C);
    return cudaGetLastError();
}

} // namespace rewl

namespace rewl {

// Window means of the saved fragments leaving walker j out (walker order), [h][W].
__global__ void k_loo_mean(State s, int j, double *out)
{
    const int w = blockIdx.x, nb = s.hi[w] - s.lo[w] + 1;
    for (int b = threadIdx.x; b < s.W; b += blockDim.x) {
        double v = 0.0;
        if (b < nb) {
            double acc = 0.0;
            for (int i = 0; i < s.m; ++i)
                if (i != j) acc = __dadd_rn(acc, s.frag[(size_t)(w * s.m + i) * s.W + b]);
            v = __ddiv_rn(acc, (double)(s.m - 1));
        }
        out[(size_t)w * s.W + b] = v;
    }
}

cudaError_t launch_loo_mean(const State &s, int j, double *out, cudaStream_t st)
{
    k_loo_mean<<<s.h, 256, 0, st>>>(s, j, out);
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
    k_jack<<<(B + 256) / 256, 256, 0, st>>>(theta, m, B, err);
    return cudaGetLastError();
}

} // namespace rewl
