// rewl_move.cuh -- the WL move kernels (Sec. 2): device code and kernel templates.  The kernels are
// instantiated in rewl_move_*.cu, one file per group so that they compile in parallel.
#pragma once
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
// One warp per walker (and a second one that draws for it, below).  Shared memory holds the lattice,
// an int64 shadow V(b) = round(ln g0(b) 2^32) + (visits) * round(ln f 2^32) of ln g over the
// window, and the proposals drawn ahead.  Moves are taken in batches of up to 32:
//   1. lane j takes the proposal of step t+j from the ring (site, neighbours, ln u, and which
//      earlier steps propose the same site or a neighbour) and evaluates its energy change on the
//      lattice as it is at the batch start;
//   2. lane x keeps the shadow of cached bin x (32 bins around the current one) in a register;
//      the cache moves when the walker nears its edge;
//   3. small ln f: lane j compares its threshold with the half-precision ratio table
//      ln g(x) - ln g(x + dk) for every cached x at once, which gives a 32-bit mask "step j is
//      surely accepted from x".  Walking the batch is then a chain of integer shifts and
//      multiply-adds on these masks, four steps at a time.  A step that is surely accepted or
//      rejected under a margin that covers every rounding and the visits since the table was
//      taken needs no more; another one is decided in float32 with those visits (at middling
//      ln f, where there are several, all lanes at once against the path just walked), and if
//      that is too close as well, on the shadow or in float64.
//      Large ln f, where each visit turns later decisions: the path is walked with running
//      float32 values through shuffles, every step screened by the same kind of margin;
//   4. the batch is cut before the first step whose site or a neighbour of it an earlier step of
//      the batch changed, and the side effects (spin flips, visits) of the steps before the cut are
//      applied lane-parallel.
// A step inside every margin is decided from the float64 values rebuilt exactly (seqadd of
// the interval-start ln g and the visit counts); at the end of the launch the float64 ln g of
// every bin is rebuilt the same way, so the state equals that of the sequential walk bit for bit.
//
// What bounds it: the dependent chain of one batch, about 1300 cycles for 29 steps at ln f = 2^-20
// on Ising L=64.  A walker is one chain and the workloads have 1-2 walkers per SM sub-partition, so
// latencies set the pace, not issue slots or memory (measured on GB300 in cycles: integer op or
// FMA 4, a predicate before use 10, shuffle 24-28, shared load 29-34, shared atomic 50, ballot
// 23, redux min 22, popc 20, ffs 42, match_any of 32 different values 375).  Hence masks and shifts
// instead of predicates, and the random numbers and conflicts, 100 instructions and four shared
// round trips a batch that need no lattice, in a second warp while the walkers of the launch leave
// warp slots free (move kernel, Ising L=64 32 x 16, ln f = 2^-20: 378 us with the drawing in the
// same warp, 259 us with a second one; 600 us with the 32-step chain of shuffles, match_any and
// predicates before).  Workloads, us per launch of 10^4 moves, that kernel -> this one: Ising L=64 32 x 16
// at 2^-20 600 -> 259, Ising L=32 8 x 8 at 2^-12 770 -> 327, Potts L=40 64 x 16 at 2^-10 810 -> 463,
// Potts L=80 64 x 16 at 2^-24 700 -> 333, at ln f = 1 730 -> 580, Ising L=8 4 x 1 1960 -> 902.
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

// visits of bin b since the launch started: the shadow grew by lnfq per visit
__device__ __forceinline__ uint32_t visits(const long long *V, const double *glng, int b, long long lnfq)
{
    return (uint32_t)((V[b] - to_fixed(glng[b])) / lnfq);
}

// ln g and H of bin b at the end of a launch: v visits since it started
__device__ __forceinline__ void write_back(double *gl, uint32_t *gH, int b, double lnf, double x, uint32_t v)
{
    if (v == 0u) return;
    if (!seqadd_in_binade(x, lnf, v, &x)) x = seqadd(x, lnf, v);
    gl[b] = x;
    gH[b] += v;
}

// Float64 decision from the exact values (rare): ln g of bins k and k' rebuilt by seqadd from
// the launch-start values and the visits recorded in the shadow.
static __device__ __noinline__ bool exact_value_decision(const double *glng, const long long *V, int lo,
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

// Margin of a decision on the shadow, in units of 2^-32: both shadow values, the float32 ln u, the
// float64 difference of ln g values below 2^31 (half an ulp, 2^-22) and the conversion of ln u
// (one unit).
__device__ __forceinline__ long long shadow_margin(double maxabs, int T, double lnf, bool frozen, double eps_l)
{
    return (long long)(2.0 * shadow_error(maxabs, T, lnf, frozen) + (eps_l + 0x1p-21) * 0x1p32) + 4;
}

// 1 / 0: accepted / rejected for sure on the shadow values, -1: too close.
__device__ __forceinline__ int shadow_decision(long long Vk, long long Vkp, uint32_t w2, long long margin)
{
    const long long e = (Vk - Vkp) - (long long)__float2ll_rz(lnu32(w2) * 0x1p32f);
    return e > margin ? 1 : (e < -margin ? 0 : -1);
}

// Ratio table: rows d = -DM .. DM of 32 half-precision differences ln g(x) - ln g(x + d) over
// the cached bins x; word w of a row holds x = w and x = w + 16.  A row is 80 bytes, so the
// 16-byte loads of eight lanes at eight different rows meet eight different bank groups.
constexpr int ROW_BYTES = 80;
constexpr int LIN_ROW = 36; // floats in a row of its float32 copy, in order of x

// ---- shared memory of one walker of the warp kernel
constexpr unsigned NO_CLAIM = 0xffu; // stamp of a site that the last drawn block does not propose

struct WalkerMem {
    uint8_t *sp;        // [N] lattice
    uint8_t *stamp;     // [N] last lane of the block drawn last that proposes the site
    long long *V;       // [W] shadow of ln g
    uint32_t *vis;      // [W bits] bin visited
    unsigned char *tab; // ratio table
    float *lin;         // the ratio table in float32, rows of LIN_ROW
    uint4 *bc;          // [24] masks and bin changes of the steps
    uint4 *trail;       // [16] what the running walk left (in place of the table)
    unsigned *cnt;      // [32] visits of the cached bins not yet in V
    uint4 *ring;        // [MOVE_RING] proposals drawn ahead
    uint32_t *near;     // [MOVE_RING] their earlier neighbours
    int *ctl;           // [4] steps drawn, steps taken, stop drawing
    __device__ __forceinline__ WalkerMem(unsigned char *base, int N, int W)
    {
        sp = base;
        stamp = sp + pad16(N);
        V = reinterpret_cast<long long *>(stamp + pad16(N));
        vis = reinterpret_cast<uint32_t *>(V + padw(W));
        tab = reinterpret_cast<unsigned char *>(vis + visw(W));
        trail = reinterpret_cast<uint4 *>(tab);
        lin = reinterpret_cast<float *>(tab + MOVE_TAB_BYTES);
        bc = reinterpret_cast<uint4 *>(lin + 9 * LIN_ROW);
        cnt = reinterpret_cast<unsigned *>(bc + 24);
        ring = reinterpret_cast<uint4 *>(cnt + 32);
        near = reinterpret_cast<uint32_t *>(ring + MOVE_RING);
        ctl = reinterpret_cast<int *>(near + MOVE_RING);
    }
};


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

// The random words of step i of a launch.
template <bool REPLAY>
__device__ __forceinline__ void draw_words(const State &s, const MoveCfg &c, int slot, unsigned long long st0, int i,
                                           uint32_t &w0, uint32_t &w1, uint32_t &w2)
{
    if (REPLAY) {
        const uint32_t *wp = c.words + ((size_t)slot * c.T + i) * 3;
        w0 = i < c.T ? wp[0] : 0u;
        w1 = i < c.T ? wp[1] : 0u;
        w2 = i < c.T ? wp[2] : 0u;
    } else {
        const unsigned long long sn = st0 + (unsigned long long)i;
        const u32x4 r = philox((uint32_t)sn, (uint32_t)(sn >> 32), (uint32_t)(s.slot0 + slot),
                               (s.inst << 8) | TAG_MOVE, s.key0, s.key1);
        w0 = r.x;
        w1 = r.y;
        w2 = r.z;
    }
}

// The block of 32 steps drawn before: each lane's site, and the lanes whose site a later lane of the block
// proposes again (their stamps are gone).
struct Drawn {
    int site = -1;
    unsigned hidden = 0u;
};

// Proposals of steps g .. g+31 (lane j: step g + j) into the ring: site, new-state draw, the four
// neighbours, ln u; and into `near` which of the 31 steps before propose the site or one of its
// neighbours: bit 32 - d for the one d steps ago.
// `stamp` holds, between calls, for every site the last lane of the block before that proposes it.
template <bool ISING, bool REPLAY>
__device__ __forceinline__ void draw_block(const State &s, const MoveCfg &c, const WalkerMem &mem, int slot,
                                           unsigned long long st0, int g, Drawn &before, int lane)
{
    uint32_t w0, w1, w2;
    draw_words<REPLAY>(s, c, slot, st0, g + lane, w0, w1, w2);
    const int site = (int)mulhi(w0, (uint32_t)s.N);
    const Lattice lat{s.L, s.N, s.magic};
    int nb[5];
    lat.nbrs(site, nb[0], nb[1], nb[2], nb[3]);
    nb[4] = site;
    const unsigned pr = ISING ? 0u : mulhi(w1, (uint32_t)(s.q - 1));
    const float lnu = lnu32(w2);
    auto meets = [&](int sl) { return sl == nb[0] || sl == nb[1] || sl == nb[2] || sl == nb[3] || sl == nb[4]; };
    unsigned near = 0u;
    // the block before: lane l there is 32 + lane - l steps ago, at most 31 for l > lane (a smaller l
    // and NO_CLAIM shift the bit out; l = lane sets bit 0, which nothing reads)
#pragma unroll
    for (int i = 0; i < 5; ++i) near |= shl_clamp(1u, (uint32_t)mem.stamp[nb[i]] - (uint32_t)lane);
    for (unsigned h = before.hidden; h; h &= h - 1) {
        const int l = __ffs(h) - 1, sl = __shfl_sync(FULL, before.site, l);
        if (l > lane && meets(sl)) near |= 1u << (l - lane);
    }
    __syncwarp();
    if (before.site >= 0) mem.stamp[before.site] = (uint8_t)NO_CLAIM;
    before.site = site;
    before.hidden = 0u;
    __syncwarp();
    mem.stamp[site] = (uint8_t)lane;
    __syncwarp();
    // two lanes on one site: make the lowest lane's stamp stand
    int own = mem.stamp[site];
    const bool twice = __any_sync(FULL, own != lane);
    if (twice) {
        for (int it = 0; it < 32; ++it) { // each pass lowers some stamp: ends within 32 passes
            const bool again = own > lane;
            __syncwarp();
            if (!__any_sync(FULL, again)) break;
            if (again) mem.stamp[site] = (uint8_t)lane;
            __syncwarp();
            own = mem.stamp[site];
        }
    }
    // this block: lane l is lane - l steps ago (l >= lane and NO_CLAIM shift the bit out)
#pragma unroll
    for (int i = 0; i < 5; ++i) near |= shl_clamp(1u, (uint32_t)(32 - lane) + mem.stamp[nb[i]]);
    if (twice) { // the later proposals of a site, in order: the last one keeps the stamp
        unsigned late = __ballot_sync(FULL, own < lane);
        while (late) {
            const int l = __ffs(late) - 1, sl = __shfl_sync(FULL, site, l);
            late &= late - 1;
            if (lane > l && meets(sl)) near |= 1u << (32 - lane + l);
            __syncwarp();
            if (lane == l) mem.stamp[site] = (uint8_t)lane;
        }
        __syncwarp();
        before.hidden = __ballot_sync(FULL, mem.stamp[site] != lane);
    }
    const int e = (g + lane) & (MOVE_RING - 1);
    mem.ring[e] = make_uint4((unsigned)site | (pr << 16), (unsigned)nb[0] | ((unsigned)nb[1] << 16),
                             (unsigned)nb[2] | ((unsigned)nb[3] << 16), __float_as_uint(lnu));
    mem.near[e] = near;
}

// Words in shared memory that two warps of a CTA hand work over with.  (A fence after a plain load
// would do the same, but holds the walker up for hundreds of cycles.)
// Every lane loads such a word itself, so that what it reads or writes afterwards comes after its own
// acquire, and the lanes then go on with the smallest value any of them saw (`agreed`): lanes of a warp
// need not load at the same instant, and a branch on different values would part them before the
// next full-mask vote.  A word is published by lane 0 after a __syncwarp, with release, so that it covers
// what all lanes did.
__device__ __forceinline__ int load_acquire(const int *p)
{
    int v;
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
    return v;
}
// the same into v where `need` holds, without a branch
__device__ __forceinline__ void poll(const int *p, int &v, bool need)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q ld.acquire.cta.shared.b32 %0, [%1];\n\t}"
                 : "+r"(v)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"((int)need)
                 : "memory");
}
__device__ __forceinline__ void store_release(int *p, int v)
{
    asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void store_relaxed(int *p, int v)
{
    asm volatile("st.relaxed.cta.shared.b32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}

__device__ __forceinline__ int agreed(int v) { return (int)__reduce_min_sync(FULL, (unsigned)v); } // v >= 0

// Polls of shared memory before a warp gives up on its partner: the first warp on the second, which
// is never long, and the second, asleep between polls, on the first, which may rebuild float64
// values for seconds (a tie in every addition of a bin's 10^8 visits).
constexpr int SPIN_LIMIT = 1 << 22, SLEEP_LIMIT = 1 << 25;
// Sleep between the drawing warp's polls.  A ring in use holds 1.5 us of late steps or more beyond the block it has
// no room for yet, so the walker does not wait for a sleeper, whose polls take issue slots.  us per launch at
// 50 / 400 / 1200 ns: Potts L=80 64 x 16 at ln f = 1 593 / 580 / 572, at 2^-24 336 / 333 / 353, Potts L=40
// 64 x 16 470 / 463 / 466, Ising L=64 32 x 16 at 2^-20 259 / 259 / 285.
constexpr unsigned DRAW_SLEEP_NS = 400;

// The second warp of a walker: draws blocks ahead of the first as the ring has room.
template <bool ISING>
__device__ __forceinline__ void draw_walker(const State &s, const MoveCfg &c, const int slot, unsigned char *base,
                                            const int lane)
{
    if (s.status != nullptr && s.status->done) return;
    const WalkerMem mem(base, s.N, s.W);
    const unsigned long long st0 = s.step[slot];
    for (int i = lane; i < (pad16(s.N) >> 2); i += 32) reinterpret_cast<uint32_t *>(mem.stamp)[i] = ~0u;
    __syncwarp();
    Drawn before;
    for (int g = 0; g < c.T + 64; g += 32) { // the first warp asks for 33 steps beyond the last
        for (int it = 0; g + 32 - agreed(load_acquire(mem.ctl + 1)) > MOVE_RING; ++it) {
            if (__any_sync(FULL, load_acquire(mem.ctl + 2) != 0) || it > SLEEP_LIMIT) return;
            __nanosleep(DRAW_SLEEP_NS);
        }
        draw_block<ISING, false>(s, c, mem, slot, st0, g, before, lane);
        __syncwarp();
        if (lane == 0) store_release(mem.ctl, g + 32);
    }
}

// How the batches of a launch are walked, by ln f: with running values; through the ratio table, the path
// verified as a whole where a step is too close for it; through the table, such steps one by one.
enum Walk { RUNNING, VERIFIED, SURE };

// One walker's `c.T` moves; `base` is the walker's shared-memory block, the whole warp calls.
// NP: pairs of steps in a batch (16, or fewer for small lattices, where sites soon repeat).
// AHEAD: another warp draws the proposals (draw_walker), else this one does.
template <bool ISING, bool REPLAY, bool CHECK, bool AHEAD, int NP, Walk WALK>
__device__ __forceinline__ void move_walker_n(const State &s, const MoveCfg &c, const int slot,
                                              unsigned char *base, const int lane)
{
    constexpr int DM = ISING ? 2 : 4; // largest |bin change| of a move
    const WalkerMem mem(base, s.N, s.W);
    uint8_t *sp = mem.sp;
    long long *V = mem.V;
    uint32_t *vis = mem.vis;
    unsigned char *tab = mem.tab;
    uint4 *bc = mem.bc, *trail = mem.trail;

    const int w = slot / s.m;
    const int lo = s.lo[w], hi = s.hi[w], nb = hi - lo + 1;
    const int kstart = s.k[slot];
    if (lo < 0 || nb < 1 || nb > s.W || kstart < lo || kstart > hi) { // malformed input: refuse
        if (lane == 0) {
            if (AHEAD) store_relaxed(mem.ctl + 2, 1);
            atomicOr(&s.status->err, ERR_INPUT);
        }
        return;
    }
    const double lnf = s.lnf[w];
    const bool frozen = s.finished[w] != 0;
    const int cfg = s.cfg ? s.cfg[slot] : slot;
    int8_t *gsp = s.spins + (size_t)cfg * s.spin_stride;
    const double *glng = s.lng + (size_t)slot * s.W;
    uint32_t *gH = s.H + (size_t)slot * s.W;
    const int T = c.T;

    // ---- load lattice, shadow ln g
    if (s.vec_spins) {
        const int4 *src = reinterpret_cast<const int4 *>(gsp);
        int4 *dst = reinterpret_cast<int4 *>(sp);
#pragma unroll 4
        for (int i = lane; i < (s.N >> 4); i += 32) dst[i] = src[i];
    } else {
#pragma unroll 4
        for (int i = lane; i < s.N; i += 32) sp[i] = (uint8_t)gsp[i];
    }
    if (!AHEAD)
        for (int i = lane; i < (pad16(s.N) >> 2); i += 32) reinterpret_cast<uint32_t *>(mem.stamp)[i] = ~0u;
    unsigned long long mxb = 0; // bits of the largest |ln g| (they order like the numbers, NaN above all)
#pragma unroll 4
    for (int b = lane; b < nb; b += 32) {
        const double x = glng[b];
        const unsigned long long ab = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
        mxb = ab > mxb ? ab : mxb;
        V[b] = ab < 0x41d0000000000000ULL ? to_fixed(x) : 0LL; // below 2^30
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(FULL, mxb, o);
        mxb = ob > mxb ? ob : mxb;
    }
    const bool bad_in = mxb >= 0x41d0000000000000ULL;
    const double mx = bad_in ? 0.0 : __longlong_as_double((long long)mxb);
    // visited bits: the bins any walker of the window had visited when this launch started,
    // the start bin, and every bin this walker enters for the first time (always through the
    // float64 path below)
    // (replay has no window mask: every bin counts as visited there)
    const uint8_t *gmask = s.mask ? s.mask + (size_t)w * s.W : nullptr;
#pragma unroll 4
    for (int i = 0; i < visw(s.W); ++i) { // word i: bins 32i .. 32i+31, one per lane
        const int b = 32 * i + lane;
        const unsigned bits = __ballot_sync(FULL, b < nb && (gmask == nullptr || gmask[b]));
        if (lane == 0) vis[i] = bits;
    }
    if (lane == 0) vis[(kstart - lo) >> 5] |= 1u << ((kstart - lo) & 31); // the start bin
    __syncwarp(); // the first cache_load reads these words
    // the shadow of a running window ends the launch below (max |ln g| + T ln f) 2^32 < 2^62,
    // and ln f 2^32 must not round to zero; a frozen window adds nothing to it
    const bool lnf_ok = frozen || (lnf >= 0x1p-32 && lnf < 0x1p20 && mx + (double)T * lnf < 0x1p30);
    if (bad_in || !lnf_ok) {
        // the int64 shadow would overflow or lose the increment: leave the state untouched
        if (lane == 0) {
            if (AHEAD) store_relaxed(mem.ctl + 2, 1);
            atomicOr(&s.status->err, ERR_RANGE);
        }
        return;
    }
    const long long lnfq = __double2ll_rn(__dmul_rn(lnf, 0x1p32));
    const long long lnfq_add = frozen ? 0LL : lnfq;
    const long long Mq = shadow_margin(mx, T, lnf, frozen, c.eps_l);
    // interval-constant part of the float32 screening margin (ln units)
    const float Mbase = (float)(c.eps_l + 2.0 * shadow_error(mx, T, lnf, frozen) * 0x1p-32) * (1.0f + 0x1p-20f) + 0x1p-21f;
    const float lnf_f = frozen ? 0.0f : (float)lnf;
    // visits after which the ratio table is taken anew
    const int table_life = lnf_f > 0.0f ? (int)fminf((WALK == VERIFIED ? VERIFIED_DRIFT : SURE_DRIFT) / lnf_f, 1e8f) : 100000000;

    const unsigned long long st0 = s.step[slot];
    unsigned int nacc = 0, nex = 0, nmis = 0; // nacc: of this lane's steps
    const unsigned below = (1u << lane) - 1u;

    // Visits are counted per cache bin in shared memory and taken over when the shadow is needed:
    // lane x those of cache bin x.
    long long Vr = 0; // shadow of the lane's cached bin
    auto settle = [&]() {
        __syncwarp();
        const unsigned v = mem.cnt[lane];
        mem.cnt[lane] = 0u;
        Vr += (long long)v * lnfq_add;
        __syncwarp();
    };
    mem.cnt[lane] = 0u;

    // ---- the cached bins: lane j holds the shadow of bin wbase + j
    int wbase = kstart - 16, x = 16; // x: cache offset of the current bin
    bool bin_ok = false, far = false;
    float Lw = 0.0f, M = 0.0f, Mx0 = -1.0f;
    int cache_age = 0; // visits since the cache was loaded
    auto cache_store = [&]() {
        settle();
        if (bin_ok) V[wbase + lane - lo] = Vr;
        __syncwarp();
    };
    auto cache_load = [&](int k) {
        wbase = k - 16;
        x = 16;
        cache_age = 0;
        Mx0 = -1.0f;
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
        settle();
        const long long ref = __shfl_sync(FULL, Vr, x);
        const long long d = Vr - ref;
        Lw = __fmaf_rn(__uint2float_rn((uint32_t)d), 0x1p-32f, (float)(int)(d >> 32));
        // bound of |Lw| over the cache: twice the largest one when the cache was loaded (the
        // current bin was another one then; non-negative floats order like their bit patterns)
        // and the visits since
        if (Mx0 < 0.0f)
            Mx0 = 2.0f * __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(bin_ok && !far ? fabsf(Lw) : 0.0f)));
        const float Mx = Mx0 + (float)(cache_age + 33) * lnf_f + 0x1p-20f;
        M = Mbase + 40.0f * ulpf(2.0f * Mx);
        if (!bin_ok) Lw = INFINITY; // a move there is rejected: ln g(k) - inf < ln u
        if (far) Lw = __int_as_float(0x7fc00000);
    };
    float *lin = mem.lin;
    if (WALK != RUNNING) { // row 0 of the table: a step that keeps the energy never moves
        reinterpret_cast<__half *>(tab + DM * ROW_BYTES)[lane] = __float2half_rn(-INFINITY);
        lin[DM * LIN_ROW + lane] = -INFINITY;
    }
    cache_load(kstart);
    int table_age = table_life + 1; // visits since the table was taken

    int g = 0; // steps drawn (as far as this warp knows), the same in every lane
    Drawn before;
    // steps up to `upto` drawn; false if the partner warp does not come
    auto drawn = [&](int upto) -> bool {
        if (AHEAD) {
            for (int it = 0; g < upto && it < SPIN_LIMIT; ++it) g = agreed(load_acquire(mem.ctl));
            return g >= upto;
        }
        while (g < upto) {
            draw_block<ISING, REPLAY>(s, c, mem, slot, st0, g, before, lane);
            g += 32;
            __syncwarp();
        }
        return true;
    };
    auto give_up = [&](int err) {
        if (lane == 0) {
            if (AHEAD) store_relaxed(mem.ctl + 2, 1);
            atomicOr(&s.status->err, err);
        }
    };
    if (!drawn(33)) {
        give_up(ERR_STALL);
        return;
    }

    int *dks = reinterpret_cast<int *>(bc + 8);       // bin changes of the steps
    unsigned *sq = reinterpret_cast<unsigned *>(bc + 16); // their acceptance masks
    const int g1 = -((lane & 3) > 0), g2 = -((lane & 3) > 1), g3 = -((lane & 3) > 2); // steps of the group before
    int t = 0;
    uint4 pe = mem.ring[lane]; // lane j: the proposal of step t + j
    uint32_t pnear = mem.near[lane];
    while (t < T) {
        const int n = min(2 * NP, T - t);
        const int site = (int)(pe.x & 0xffffu);
        const unsigned c1 = sp[pe.y & 0xffffu], c2 = sp[pe.y >> 16], c3 = sp[pe.z & 0xffffu], c4 = sp[pe.z >> 16];
        const uint32_t s0 = sp[site];
        // earlier lanes that propose this site or one of its neighbours; settled after the walk: the
        // batch ends before the first step one of whose claims was accepted
        const unsigned claims = lane ? pnear >> (32 - lane) : 0u;
        const int cut = lane >= n ? -1 : 0;
        const uint32_t nbytes = __byte_perm(__byte_perm(c1, c2, 0x0040), __byte_perm(c3, c4, 0x0040), 0x5410);
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
        // a proposal that keeps the energy is always accepted and keeps the bin: the walk sees a
        // sure non-move, the lane itself records the flip
        const bool dz = dk == 0;
        const float lnu = __uint_as_float(pe.w);
        dks[lane] = dk;

        // ---- the walk: cache offsets xb, xa of the bin before and after step `lane`.  The batch
        // stops before step `stop`; `open` says that this step is not decided yet.
        int xb, xa, stop, scr = -1;
        bool open;
        auto stop_at = [&](bool accepted, int sure) {
            const unsigned met = claims & __ballot_sync(FULL, accepted);
            const int end = cut | sign_mask((int)(met | (0u - met)));
            const unsigned v = __reduce_min_sync(FULL, (unsigned)pick(end, 2 * lane, pick(sure, 64, 2 * lane + 1)));
            stop = (int)(v >> 1);
            open = v & 1u;
        };
        const bool edge = (unsigned)(x - CACHE_LO) > (unsigned)(CACHE_HI - CACHE_LO);
        if (__builtin_expect(edge, 0)) { // the current bin near the edge of the cache: cache the bins around it
            const int k = wbase + x;
            cache_store();
            cache_load(k);
        }
        if (WALK != RUNNING) {
            if (__builtin_expect(edge || table_age > table_life, 0)) { // rows of the ratio table
                cache_floats();
#pragma unroll
                for (int d = 1; d <= DM; ++d) {
                    float up = __shfl_down_sync(FULL, Lw, d);
                    if (lane + d > 31) up = __int_as_float(0x7fc00000);
                    const float D = Lw - up;
                    const __half h = __float2half_rn(D);
                    const int xd = (lane + d) & 31;
                    *reinterpret_cast<__half *>(tab + (DM + d) * ROW_BYTES + 4 * (lane & 15) + 2 * (lane >> 4)) = h;
                    *reinterpret_cast<__half *>(tab + (DM - d) * ROW_BYTES + 4 * (xd & 15) + 2 * (xd >> 4)) = __hneg(h);
                    lin[(DM + d) * LIN_ROW + lane] = D;
                    lin[(DM - d) * LIN_ROW + xd] = -D;
                }
                table_age = 0;
                __syncwarp();
            }
            // the step is surely accepted from bin offset x if D(x) > tA, surely rejected if
            // D(x) < tR, whatever the visits since the table was taken did to ln g.  The walk takes
            // what is not sure for a rejection (VERIFIED: for what the table says).
            const float mg = __fmaf_rn((float)(table_age + lane + 1), lnf_f, M);
            const __half2 tS = __float2half2_rn(WALK == VERIFIED ? lnu : lnu + mg);
            const float tR = lnu - mg, tA = lnu + mg;
            const uint4 *row = reinterpret_cast<const uint4 *>(tab + dkm * ROW_BYTES);
            const float *lrow = lin + dkm * LIN_ROW;
            unsigned S4[4]; // one a load, so that the chain is short
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const uint4 qv = row[v];
                const uint32_t ww[4] = {qv.x, qv.y, qv.z, qv.w};
                S4[v] = 0u;
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    S4[v] |= __hgt2_mask(*reinterpret_cast<const __half2 *>(&ww[e]), tS) & (0x00010001u << (4 * v + e));
            }
            unsigned S = (S4[0] | S4[1]) | (S4[2] | S4[3]); // bit x: accepted from x
            int known = 0; // -1: step `lane` was decided below
            int4 d;        // of the lane's group of four steps: bin changes
            uint4 q;       // and masks: from bin offset x at the start of the group, step i of it
                           // moves if bit x of mask i is set, whatever the steps before it do
            auto walk = [&]() {
                sq[lane] = S;
                __syncwarp();
                q = reinterpret_cast<const uint4 *>(sq)[lane >> 2];
                d = reinterpret_cast<const int4 *>(dks)[lane >> 2];
                // bit x of `seen(Q, e)`: bit x + e of Q, |e| <= 8
                auto seen = [](unsigned Q, int e) { return (int)__funnelshift_r(Q << 8, Q >> 24, (unsigned)(8 + e)); };
                q.y = (unsigned)pick((int)q.x, seen(q.y, d.x), (int)q.y);
                q.w = (unsigned)pick((int)q.z, seen(q.w, d.z), (int)q.w);
                const unsigned m2 = q.z, m3 = q.w; // the second pair's, from where the first leaves x
                q.z = (unsigned)pick((int)q.x, pick((int)q.y, seen(m2, d.x + d.y), seen(m2, d.x)),
                                     pick((int)q.y, seen(m2, d.y), (int)m2));
                q.w = (unsigned)pick((int)q.x, pick((int)q.y, seen(m3, d.x + d.y), seen(m3, d.x)),
                                     pick((int)q.y, seen(m3, d.y), (int)m3));
                if (!(lane & 3)) bc[lane >> 2] = q;
                __syncwarp();
                int y = 31 - x; // mask << y has the bit of offset x on top
                unsigned pk[2] = {0u, 0u};
#pragma unroll
                for (int p = 0; p < NP / 2; ++p) {
                    const uint4 a = bc[p];
                    const int4 e = reinterpret_cast<const int4 *>(dks)[p];
                    pk[p >> 2] |= (unsigned)y << (8 * (p & 3));
                    const int u = sign_mask((int)(a.x << y)) * e.x + y, v = sign_mask((int)(a.y << y)) * e.y;
                    y = (sign_mask((int)(a.z << y)) * e.z + u) + (sign_mask((int)(a.w << y)) * e.w + v);
                }
                int yb = (int)(((lane < 16 ? pk[0] : pk[1]) >> (8 * ((lane >> 2) & 3))) & 31u);
                yb += (sign_mask((int)(q.x << yb)) & g1) * d.x + (sign_mask((int)(q.y << yb)) & g2) * d.y +
                      (sign_mask((int)(q.z << yb)) & g3) * d.z;
                xb = 31 - yb;
                const int mv = sign_mask((int)(S << yb));
                xa = xb + (mv & dk);
                int sure;
                if (WALK == VERIFIED) {
                    const float D = lrow[xb];
                    sure = pick(mv, sign_mask(__float_as_int(tA - D)), sign_mask(__float_as_int(D - tR)));
                } else {
                    sure = mv | known | sign_mask(__float_as_int(lrow[xb] - tR));
                }
                if (CHECK) sure = dz || (unsigned)(xb + dk - (lo - wbase)) >= (unsigned)nb ? -1 : 0;
                stop_at(dz || mv != 0, sure);
            };
            walk();
            bool fresh = table_age == 0;
            while (__builtin_expect(open, 0)) {
                if (WALK == VERIFIED) {
                    if ((unsigned)__shfl_sync(FULL, xb + dk, stop) >= 32u) {
                        open = stop == 0; // else the next batch's cache will hold the target
                        break;
                    }
                    if (!fresh) { // bring the cached values up to date
                        const float Mt = M;
                        cache_floats();
                        M = fmaxf(M, Mt);
                        fresh = true;
                    }
                    // Some step is too close for the table.  Every lane takes its own step's ln g
                    // difference with the visits on the path before it, in float32; the path is right
                    // as far as all of them agree with it.  The first one that does not is put right
                    // and the walk taken again.
                    const int xt = xb + dk;
                    unsigned at = below, to = below; // steps before this one that ended in xb, in xt
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const unsigned b = __ballot_sync(FULL, (xa >> i) & 1);
                        at &= ((xb >> i) & 1) ? b : ~b;
                        to &= ((xt >> i) & 1) ? b : ~b;
                    }
                    const bool out = (unsigned)xt >= 32u;
                    const float Lb = __shfl_sync(FULL, Lw, xb), Lt = __shfl_sync(FULL, Lw, xt);
                    const float e = out ? __int_as_float(0x7fc00000)
                                        : __fmaf_rn((float)(__popc(at) - __popc(to)), lnf_f, Lb - Lt) - lnu;
                    if (CHECK) {
                        const float D = lrow[xb];
                        scr = __shfl_sync(FULL, D > tA ? 1 : (D < tR ? 0 : (e > M ? 1 : (e < -M ? 0 : -1))), stop);
                        break;
                    }
                    stop_at(dz || xa != xb, dz || (xa != xb ? e > M : e < -M) ? -1 : 0);
                    if (!open) break;
                    const int v = __shfl_sync(FULL, e > M ? 1 : (e < -M ? 0 : (out ? 2 : 3)), stop);
                    if (v >= 2) { // outside the cache as above, or too close: float64
                        open = stop == 0 || v == 3;
                        break;
                    }
                    if (lane == stop) S = (S & ~(1u << xb)) | ((unsigned)v << xb);
                } else {
                    // step `stop`: its ln g difference with the visits before it, in float32
                    const int u = stop;
                    const int xu = __shfl_sync(FULL, xb, u), du = __shfl_sync(FULL, dk, u);
                    const int xt = xu + du;
                    if ((unsigned)xt >= 32u) {
                        open = u == 0; // else the next batch's cache will hold the target
                        break;
                    }
                    if (!fresh) { // bring the cached values up to date
                        const float Mt = M;
                        cache_floats();
                        M = fmaxf(M, Mt);
                        fresh = true;
                    }
                    const unsigned bu = (1u << u) - 1u;
                    const int cx = __popc(__ballot_sync(FULL, xa == xu) & bu), ct = __popc(__ballot_sync(FULL, xa == xt) & bu);
                    const float e = __fmaf_rn((float)(cx - ct), lnf_f, __shfl_sync(FULL, Lw, xu) - __shfl_sync(FULL, Lw, xt)) -
                                    __shfl_sync(FULL, lnu, u);
                    if (CHECK) {
                        const int sure = ((S >> xu) & 1u) ? 1 : (lrow[xu] < tR ? 0 : -1);
                        scr = __shfl_sync(FULL, sure, u);
                        if (scr < 0) scr = e > M ? 1 : (e < -M ? 0 : -1);
                        break;
                    }
                    if (!(fabsf(e) > M)) break; // too close: float64
                    if (lane == u) {
                        known = -1;
                        if (e > M) S |= 1u << xu;
                    }
                }
                walk();
            }
            table_age += stop;
        } else {
            // Large ln f: the visits of the batch decide its later steps, so the path is walked
            // with running float32 values.  Steps are resolved in pairs: the three cache
            // lookups a pair can need (k' of the first step; k' of the second after the first
            // moved / stayed) are issued together and the second step is evaluated in both
            // worlds, so one shuffle latency covers two moves.  Decision variable:
            // v = M - (ln g(k) - ln g(k') - ln u); accept if v < 0, reject if v > 2M, else unsure.
            // A target outside the 32 cached bins reads a wrong lane; such steps are found after
            // the loop and cut there as well.
            // Steps that keep the energy never move: only the others are walked, each with the ln f of
            // the visits such steps made since the one before it (G).
            cache_floats();
            const unsigned act = __ballot_sync(FULL, !dz && lane < n), earlier = act & below;
            const int rank = __popc(earlier), nact = __popc(act);
            float2 *gap = reinterpret_cast<float2 *>(bc + 16);
            if (!dz) {
                reinterpret_cast<uint2 *>(bc)[rank] = make_uint2(__float_as_uint(lnu + M), (unsigned)dk);
                reinterpret_cast<float *>(gap)[rank] = (float)(lane - 32 + __clz(earlier)) * lnf_f;
            }
            __syncwarp();
            float Lr = Lw;   // the cache, with the running values of the bins left
            int xk = x;      // cache offset of the current bin
            float Lk = 0.0f; // its running value (the cache holds it only once left)
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                if ((p & 1) == 0 && p > 0 && 2 * p >= nact) break; // (what is behind nact is not read)
                const uint4 a = bc[p];
                const float2 G = gap[p];
                const int d0 = (int)a.y, d1 = (int)a.w;
                const int x0 = xk + d0; // k' of step i
                const int xA = x0 + d1; // k' of step i+1 if step i moved
                const int xR = xk + d1; // k' of step i+1 if step i stayed
                const float L0 = __shfl_sync(FULL, Lr, x0);
                const float LA_ = __shfl_sync(FULL, Lr, xA);
                const float LR = __shfl_sync(FULL, Lr, xR);
                Lk += G.x;
                const float LA = (d1 == -d0) ? Lk : LA_; // back to the bin just left
                const int onk = lane == xk ? -1 : 0, on0 = lane == x0 ? -1 : 0;
                const float G1 = lnf_f + G.y;  // step i's visit and those before step i+1
                const float Ls = Lk + G1;      // value before step i+1 if step i stayed
                const float Lm = L0 + G1;      // value before step i+1 if step i moved
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
            const uint2 *walked = reinterpret_cast<const uint2 *>(trail);
            xb = rank ? (int)walked[rank - 1].x : x;
            const uint2 tr = walked[rank & 31];
            xa = dz ? xb : (int)tr.x;
            const float v = __uint_as_float(tr.y);
            const bool oob = (unsigned)(xb + dk) >= 32u;
            const float M2 = 2.0f * M * (1.0f + 0x1p-20f);
            bool ok = dz || ((v < 0.0f || v > M2) && !oob);
            if (CHECK) ok = dz || (unsigned)(xb + dk - (lo - wbase)) >= (unsigned)nb;
            stop_at(dz || xa != xb, ok ? -1 : 0);
            if (open) {
                const bool out = __shfl_sync(FULL, oob ? 1 : 0, stop);
                if (CHECK) {
                    const float vu = __shfl_sync(FULL, v, stop);
                    scr = out ? -1 : (vu < 0.0f ? 1 : (vu > M2 ? 0 : -1));
                } else if (stop > 0 && out) {
                    open = false; // the next batch's cache will hold the target
                }
            }
        }

        // ---- side effects of steps 0 .. stop-1
        const bool mine = lane < stop;
        const bool accj = dz || xa != xb; // step j accepted (a move to another bin, or dE = 0)
        if (mine && accj) sp[site] = (uint8_t)snew; // distinct sites: an accepted claim ends the batch
        if (mine) atomicAdd(&mem.cnt[xa], 1u);
        if (REPLAY && mine) {
            c.acc_out[(size_t)slot * T + t + lane] = accj ? 1 : 0;
            c.dk_out[(size_t)slot * T + t + lane] = dk;
        }
        cache_age += stop;
        t += stop;
        if (AHEAD) {
            poll(mem.ctl, g, g < t + 33);
            g = agreed(g);
        }
        pe = mem.ring[(t + lane) & (MOVE_RING - 1)]; // where g < t + 33 perhaps not written yet: read again below
        pnear = mem.near[(t + lane) & (MOVE_RING - 1)];
        nacc += mine && accj ? 1u : 0u;
        const int xlast = __shfl_sync(FULL, xa, stop - 1);
        x = stop > 0 ? xlast : x;
        __syncwarp();
        if (AHEAD && lane == 0) store_release(mem.ctl + 1, t);

        if (__builtin_expect(open || stop == 0 || t >= T || g < t + 33, 0)) {
            if (!open && stop == 0) { // no step done and none to decide: cannot happen (lane 0 is never cut)
                give_up(ERR_INPUT);
                return;
            }
            // a proposal too close to call in float32: decide it from the float64 values
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
                    draw_words<REPLAY>(s, c, slot, st0, t, w0, w1, w2i);
                    // the shadow settles most of them (bins seen for the first time, cached values
                    // far apart); the float64 values, thousands of cycles, the others
                    const int sd = shadow_decision(V[k - lo], V[kp - lo], w2i, Mq);
                    if (scr < 0) scr = sd;
                    acc = sd == 1;
                    if (CHECK || sd < 0) acc = exact_value_decision(glng, V, lo, k, kp, lnf, lnfq, frozen, w2i);
                    if (scr < 0) ++nex;
                    else if (CHECK && (int)acc != scr) ++nmis;
                }
                __syncwarp();
                if (acc) {
                    k = kp;
                    if (lane == 0) {
                        sp[sitei] = (uint8_t)snewi;
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
                __syncwarp();
                cache_load(k);
                table_age = table_life + 1;
            }
            if (t < T) {
                if (!drawn(t + 33)) {
                    give_up(ERR_STALL);
                    return;
                }
                pe = mem.ring[(t + lane) & (MOVE_RING - 1)];
                pnear = mem.near[(t + lane) & (MOVE_RING - 1)];
            }
        }
    }
    cache_store();

    // ---- write back lattice, float64 ln g (rebuilt exactly), H, counters
    if (s.vec_spins) {
        const int4 *src = reinterpret_cast<const int4 *>(sp);
        int4 *dst = reinterpret_cast<int4 *>(gsp);
        for (int i = lane; i < (s.N >> 4); i += 32) dst[i] = src[i];
    } else {
        for (int i = lane; i < s.N; i += 32) gsp[i] = (int8_t)sp[i];
    }
    if (!frozen) {
        double *gl = s.lng + (size_t)slot * s.W;
        const ExactDiv by(lnfq);
#pragma unroll 1
        for (int b = lane; b < nb; b += 32) {
            const double x = gl[b];
            write_back(gl, gH, b, lnf, x, by(V[b] - to_fixed(x)));
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

template <bool ISING, bool REPLAY, bool CHECK, bool AHEAD>
__device__ __forceinline__ void move_walker(const State &s, const MoveCfg &c, const int slot,
                                            unsigned char *base, const int lane)
{
    if (s.status != nullptr && s.status->done) return;
    const int w = slot / s.m;
    const double lnf = s.finished[w] ? 0.0 : s.lnf[w];
#define REWL_WALK(NP)                                                                            \
    do {                                                                                         \
        if (lnf <= (double)SURE_WALK_LNF)                                                        \
            move_walker_n<ISING, REPLAY, CHECK, AHEAD, NP, SURE>(s, c, slot, base, lane);        \
        else if (lnf <= (double)TABLE_WALK_LNF)                                                  \
            move_walker_n<ISING, REPLAY, CHECK, AHEAD, NP, VERIFIED>(s, c, slot, base, lane);    \
        else                                                                                     \
            move_walker_n<ISING, REPLAY, CHECK, AHEAD, NP, RUNNING>(s, c, slot, base, lane);     \
    } while (0)
    if (s.N >= BATCH32_SITES) REWL_WALK(16);
    else if (s.N >= BATCH16_SITES) REWL_WALK(8);
    else REWL_WALK(4);
#undef REWL_WALK
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
        V[b] = bad ? 0LL : to_fixed(x);
    }
    const bool lnf_ok = frozen || (lnf >= 0x1p-32 && lnf < 0x1p20 && mx + (double)T * lnf < 0x1p30);
    if (bad || !lnf_ok) {
        atomicOr(&s.status->err, ERR_RANGE);
        return;
    }
    const long long lnfq = frozen ? 0LL : __double2ll_rn(__dmul_rn(lnf, 0x1p32));
    const long long Mq = shadow_margin(mx, T, lnf, frozen, c.eps_l);
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
            const int scr = shadow_decision(Vk, V[kp - lo], w2, Mq);
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
    if (!frozen) {
        const ExactDiv by(lnfq);
        for (int b = 0; b < nb; ++b) {
            const double x = glng[b];
            write_back(glng, gH, b, lnf, x, by(V[b] - to_fixed(x)));
        }
    }
    s.k[slot] = k;
    s.step[slot] = st0 + (unsigned long long)T;
    s.acc[slot] += nacc;
    if (nex) atomicAdd(&s.status->n_exact, (unsigned long long)nex);
    if (nmis) atomicAdd(&s.status->n_mismatch, (unsigned long long)nmis);
}

// Warps 0 .. G-1 of a CTA move its G walkers; with AHEAD, warps G .. 2G-1 draw their proposals.
template <bool ISING, bool REPLAY, bool CHECK, bool AHEAD>
__global__ void __launch_bounds__(512, 1) k_move(State s, MoveCfg c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, G = c.walkers_per_block;
    const bool draws = AHEAD && warp >= G;
    const int wib = draws ? warp - G : warp;
    const int slot = blockIdx.x * G + wib;
    unsigned char *base = smem + (size_t)wib * move_smem_per_walker(s.N, s.W);
    if (AHEAD) {
        if (!draws && lane < 4) WalkerMem(base, s.N, s.W).ctl[lane] = 0;
        __syncthreads();
    }
    if (slot >= s.nw) return;
    if (draws) draw_walker<ISING>(s, c, slot, base, lane);
    else move_walker<ISING, REPLAY, CHECK, AHEAD>(s, c, slot, base, lane);
}

// Batched instances in one launch: CTA b serves walkers jobs[b].y .. jobs[b].y + jobs[b].z - 1 of
// instance jobs[b].x & 0xffffff, one warp per walker, or one thread per walker when bit 24 of
// jobs[b].x is set; the model and the layout are chosen per CTA.
template <bool CHECK, bool AHEAD>
__global__ void __launch_bounds__(512, 1) k_move_batch(const State *__restrict__ states,
                                                    const int4 *__restrict__ jobs, MoveCfg c)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
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
    const bool draws = AHEAD && warp >= c.walkers_per_block;
    const int wib = draws ? warp - c.walkers_per_block : warp;
    unsigned char *base = smem + (size_t)wib * move_smem_per_walker(s.N, s.W);
    if (AHEAD) {
        if (!draws && wib < job.z && lane < 4) WalkerMem(base, s.N, s.W).ctl[lane] = 0;
        __syncthreads();
    }
    if (wib >= job.z) return;
    if (draws) {
        if (s.model == 0) draw_walker<true>(s, c, job.y + wib, base, lane);
        else draw_walker<false>(s, c, job.y + wib, base, lane);
        return;
    }
    if (s.model == 0) move_walker<true, false, CHECK, AHEAD>(s, c, job.y + wib, base, lane);
    else move_walker<false, false, CHECK, AHEAD>(s, c, job.y + wib, base, lane);
}

// Launch of one instance of k_move / k_move_batch (instantiated in rewl_move_*.cu).
template <bool ISING, bool REPLAY, bool CHECK, bool AHEAD>
cudaError_t start_move(const State &s, const MoveCfg &c, int grid, size_t smem, cudaStream_t st);
template <bool CHECK, bool AHEAD>
cudaError_t start_move_batch(const State *states, const int4 *jobs, int njobs, size_t smem, const MoveCfg &c,
                             cudaStream_t st);

} // namespace rewl
