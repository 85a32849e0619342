// rewl_kernels.cuh -- kernel argument blocks and launchers shared by the host runtime.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace rewl {

// Device-side run status (one per handle).
struct DevStatus {
    long long round;              // rounds completed
    int done;                     // every window finished
    int err;                      // ERR_* bits
    unsigned long long n_exact;   // moves decided by the float64 path
    unsigned long long n_mismatch;// check_all: screen decisions that disagreed (must stay 0)
};
enum : int { ERR_PREP = 1, ERR_RANGE = 2, ERR_INPUT = 4, ERR_STALL = 8 };
constexpr int MAX_M = 1024; // walkers per window (exchange permutation in shared memory)
constexpr size_t MAX_SMEM_PER_CTA = 227u * 1024u;

// Per-walker-slot state of one REWL instance, all device pointers.
struct State {
    int model, q, L, N, nw, m, h, W, spin_stride;
    int vec_spins;            // lattices 16-byte aligned with N % 16 == 0: int4 copies
    uint32_t magic;           // ceil(2^32 / L)
    int8_t *spins;            // [nw][spin_stride] lattices (owned by configuration index)
    int *cfg;                 // [nw] slot -> configuration index
    int *k;                   // [nw] current bin of the slot's configuration
    double *lng;              // [nw][W] window-local ln g
    uint32_t *H;              // [nw][W]
    unsigned long long *step; // [nw]
    unsigned long long *acc;  // [nw]
    unsigned long long *pstep;// [nw]
    int *restarts;            // [nw]
    uint8_t *flat;            // [nw]
    const int *lo, *hi;       // [h]
    double *lnf;              // [h]
    int *iter;                // [h]
    uint8_t *finished;        // [h]
    uint8_t *mask;            // [h][W]
    unsigned long long *swap_att, *swap_acc; // [h]
    long long *it1_round;     // [h] rounds done when the first iteration ended (0: not yet)
    uint8_t *mode;            // [h] 0: ln f halving, 1: ln f = 1/t
    int schedule;             // 0: halving only, 1: switch to 1/t
    double *frag;             // [nw][W] ln g of each walker just before its window's last average
    uint32_t *hem;            // [h][W][N+1] (bin, up spins) counts, nullptr: not measured
    int production;           // rounds continue after every window finished
    DevStatus *status;
    unsigned *sync;           // [(h+1)/2 + 1] arrival counters of k_round_tail, zero between launches
    uint32_t key0, key1, inst;
    int w0, slot0;            // window-sharded run: global index of window 0 / walker slot 0
};

struct MoveCfg {
    int T;                  // attempts per walker in this launch
    int walkers_per_block;  // walkers per CTA (warps, or threads with layout 1)
    int layout;             // 0: one warp per walker, 1: one thread per walker
    int check_all;
    int ahead;              // a second warp per walker draws its proposals
    double eps_l;
    const uint32_t *words;  // replay: [nw][T][3], else nullptr (Philox)
    int *acc_out, *dk_out;  // replay: [nw][T]
};

// 32-bit words of the per-walker visited-bin bit set (padded to 16 bytes)
__host__ __device__ inline int visw(int W) { return (((W + 31) >> 5) + 3) & ~3; }

// Scratch of one walker's batch: the ratio table (9 rows of 80 bytes, and 9 of 36 floats), masks and
// bin changes of the steps, visit counts of the cached bins, the ring of proposals drawn ahead and
// four control words.
constexpr int MOVE_TAB_BYTES = 9 * 80;
constexpr int MOVE_RING = 128;
constexpr int MOVE_SCRATCH_BYTES = MOVE_TAB_BYTES + 9 * 36 * 4 + 24 * 16 + 32 * 4 + MOVE_RING * 20 + 16;
// Largest ln f at which a batch is walked through the ratio table.  Above it the visits of the batch
// itself leave too many steps undecided (us per launch, table / running walk, at 1, 1.2, 1.49 and 2 times 2^-6:
// Potts L=80 64 x 16 541 / 569, 558 / 572, 578 / 571, 606 / 573; Ising L=64 32 x 16 424 / 440, 436 / 440,
// 453 / 443, 476 / 443; Ising L=32 8 x 8 425 / 497, 440 / 496, 456 / 496, 482 / 499).
constexpr float TABLE_WALK_LNF = 0x1.8p-6f;
// Largest ln f at which undecided steps are rare enough to be taken one by one: verifying the whole path
// costs the walk registers (Potts L=40 at 2^-10: 490 us one by one, 474 verified, Ising L=64 at 2^-8 433
// and 364; at 2^-14 L=8 .. 16 gain 2 % without, at 2^-12 the two are equal).
constexpr float SURE_WALK_LNF = 0x1p-13f;
// Growth of ln g (visits x ln f) after which the ratio table is taken anew: taking it costs about 300
// cycles, a step left undecided about as much verified and twice that one by one (us per launch at
// 2^-10 / 2^-6 / 2^-4: Ising L=32 8 x 8 at ln f = 2^-12 372 / 341 / 363, Ising L=8 whole run 1099 / 954 /
// 936; Potts L=40 at 2^-10, verified, 2^-6 / 2^-5: 485 / 474).
constexpr float SURE_DRIFT = 0x1p-6f, VERIFIED_DRIFT = 0x1p-5f;
// Cache offsets of the current bin between which the cached bins stay (8 .. 23: 1 % slower; a step
// changes the bin by 4 at most).
constexpr int CACHE_LO = 6, CACHE_HI = 25;
// Smallest lattices whose batches are 32 and 16 steps (smaller ones: 8).  Sites soon repeat on a
// small lattice: a batch ends after about 5 steps on 64 sites, 13 on 256, 24 on 1024.  us per launch of Ising
// 8 x 8 at ln f = 1 / 2^-9 / 2^-20: 32 steps against 16 on L=21 730 / 533 / 429 and 631 / 534 / 422, on
// L=22 711 / 482 / 400 and 621 / 504 / 406, on L=28 586 / 363 / 291 and 575 / 442 / 356; 16 steps against 8 on
// L=9 1193 / 943 / 833 and 1051 / 935 / 829, on L=10 1083 / 865 / 750 and 988 / 884 / 774.
constexpr int BATCH32_SITES = 450, BATCH16_SITES = 100;

// Shared memory of one walker in the move kernel: lattice and stamps (a byte each per site, padded
// to 16 sites), int64 ln g shadow over the window (padded to 4 bins; the visit counts are recovered
// from it), the visited-bin bit set, the batch scratch.
__host__ __device__ inline size_t move_smem_per_walker(int N, int W)
{
    return 2u * (size_t)((N + 15) & ~15) + (size_t)((W + 3) & ~3) * 8u + (size_t)visw(W) * 4u +
           (size_t)MOVE_SCRATCH_BYTES;
}
// Whether a second warp per walker pays: it takes the drawing off the walker's chain, as long as
// all walkers of the launch are still resident at once (128 registers: 16 warps per SM).  us per launch, with
// and without it, Ising L=64 at 2^-20: 512 walkers 253 / 373, 1216 (8 per SM) 328 / 423, 1280 476 / 466; at
// ln f = 1 460 / 582, 590 / 665, 942 / 807; Potts L=20 at 2^-20 1216 walkers 633 / 771, 1280 936 / 876.
inline bool draw_ahead_pays(long long walkers, int sms, int walkers_per_cta, size_t smem_per_walker)
{
    const long long fit = (long long)(MAX_SMEM_PER_CTA / smem_per_walker);
    return walkers_per_cta <= 8 && walkers <= sms * (fit < 8 ? fit : 8);
}
// The largest lattice and window accepted: 3 bytes per site and 8 per bin within one CTA.  It leaves the batch
// scratch out, so it covers move_smem_per_walker only for rows no wider than a lattice has bins
// (W <= 2N + 1, as in every handle); a replay's wider rows run one thread per walker (replay_layout).
__host__ __device__ inline bool move_fits(int N, int W)
{
    return (size_t)((N + 15) & ~15) + (size_t)((W + 3) & ~3) * 8u + (size_t)visw(W) * 4u +
               (size_t)((N + 7) & ~7) * 2u <=
           MAX_SMEM_PER_CTA;
}
// Shared memory of one walker in the prep kernel: a 16-bit cell per site.
__host__ __device__ inline size_t prep_smem_per_walker(int N) { return 2u * (size_t)((N + 15) & ~15); }
// Shared memory of one walker of the thread-per-walker layout: lattice (16-byte padded) and the
// int64 ln g shadow over the window (padded to 2 bins, 16 bytes).
__host__ __device__ inline size_t move_smem_per_thread_walker(int N, int W)
{
    return (size_t)((N + 15) & ~15) + (size_t)((W + 1) & ~1) * 8u;
}
cudaError_t launch_move(const State &s, const MoveCfg &c, cudaStream_t st);
// Batched instances: states/jobs/tables are device arrays (see the kernels).
cudaError_t launch_move_batch(const State *states, const int4 *jobs, int njobs, size_t smem, const MoveCfg &c,
                              cudaStream_t st);
cudaError_t launch_round_tail_batch(const State *states, const int2 *tab, int n, const double2 *prm,
                                    cudaStream_t st);
cudaError_t launch_init_prep(const State &s, long long prep_budget, cudaStream_t st);
cudaError_t launch_round_tail(const State &s, double flatness, double lnf_final, cudaStream_t st);
cudaError_t launch_set_done(const State &s, cudaStream_t st);
// joint density of states g(E, M) (rewl_em.cu)
cudaError_t launch_measure_em(const State &s, cudaStream_t st);
// lattices of slots first .. first+n-1
cudaError_t launch_gather_spins(const State &s, int first, int n, int8_t *out /*[n][N]*/, cudaStream_t st);
cudaError_t launch_window_mean(const State &s, double *out /*[h][W]*/, cudaStream_t st);
// n joins at once: of the window means at mean + r h W, r = 0 .. n-1
cudaError_t launch_stitch(const State &s, int n, const double *mean, double de, int step, int norm,
                          double target, double *out /*[n][B+1]*/, int *joins /*[n][h]*/, double *at /*[n][h][2]*/,
                          int *ok /*[n]*/, int B, cudaStream_t st);

// window-sharded runs: the exchange of the pair across a shard boundary (Eq. 1), in four steps
// (side 1: this shard holds the pair's lower window, its last; side 0: the upper, its first)
cudaError_t launch_bnd_bins(const State &s, int side, int *bins, cudaStream_t st);
cudaError_t launch_bnd_half(const State &s, int side, int plo, int phi, const int *pbins,
                            double *half, cudaStream_t st);
cudaError_t launch_bnd_decide(const State &s, int side, const double *half, const double *phalf,
                              uint8_t *acc, int8_t *lat_out, cudaStream_t st);
cudaError_t launch_bnd_import(const State &s, int side, const int *pbins, const uint8_t *acc,
                              const int8_t *plat, cudaStream_t st);
// the n means that leave out walkers j0 .. j0+n-1
cudaError_t launch_loo_mean(const State &s, int j0, int n, double *out /*[n][h][W]*/, cudaStream_t st);
cudaError_t launch_jack(const double *theta /*[m][B+1]*/, int m, int B, double *err, cudaStream_t st);
cudaError_t launch_thermo(const double *lng, int model, int L, const double *T, int nT, double *U,
                          double *C, cudaStream_t st);
cudaError_t launch_philox(const uint32_t *ctr, const uint32_t *key, uint32_t *out, int n,
                          cudaStream_t st);
cudaError_t launch_lnu(const uint32_t *w, double *out, int n, cudaStream_t st);
cudaError_t launch_lnu_bound(uint64_t begin, uint64_t end, double *max_err,
                             unsigned long long *n_bad, cudaStream_t st);
cudaError_t launch_seqadd(const double *x, const double *f, const uint32_t *c, double *out,
                          int n, cudaStream_t st);

} // namespace rewl
