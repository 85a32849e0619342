// rewl_mlp.cu -- the warm-start network: a 3 -> 64 -> 64 -> 1 MLP (tanh, float32) that maps
// (e = E/N in the Potts convention, q, 1/L) to ln g(E)/N, trained on converged REWL results of
// small lattices and evaluated for a larger one.  Forward, backward (mean squared error),
// a fixed-order gradient reduction (results do not depend on scheduling) and Adam.
//
// Parameter vector (4481 floats): W1[64][3], b1[64], W2[64][64] (W2[i][j]: hidden-1 unit j ->
// hidden-2 unit i), b2[64], W3[64], b3.
//
// Sizes are tiny (a 64x64 layer over ~10^4 samples) and the weights are float32, so CUDA cores are
// used: a step is a few microseconds of FMA, and a tensor-core product would round its operands.
#include <cmath>
#include <cstdint>
#include <string>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "rewl.h"
#include "rewl_device.cuh"

namespace {

constexpr int HID = 64;
constexpr int OFF_W1 = 0, OFF_B1 = HID * 3, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID,
              OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID, NPARAM = OFF_B3 + 1;
static_assert(NPARAM == REWL_MLP_NPARAM, "parameter count");
constexpr int TILE = 128; // samples per CTA in the gradient kernel

thread_local std::string g_mlp_err;

__device__ __forceinline__ void load_params(const float *__restrict__ P, float *sP)
{
    for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) sP[i] = P[i];
    __syncthreads();
}

// forward of one sample; h1, h2 receive the hidden activations
__device__ __forceinline__ float mlp_fwd1(const float *sP, float x0, float x1, float x2,
                                          float *h1, float *h2)
{
#pragma unroll 8
    for (int j = 0; j < HID; ++j) {
        const float z = sP[OFF_B1 + j] + sP[OFF_W1 + 3 * j] * x0 + sP[OFF_W1 + 3 * j + 1] * x1 +
                        sP[OFF_W1 + 3 * j + 2] * x2;
        h1[j] = tanhf(z);
    }
    float y = sP[OFF_B3];
    for (int i = 0; i < HID; ++i) {
        float z = sP[OFF_B2 + i];
        const float *w = sP + OFF_W2 + HID * i;
#pragma unroll 16
        for (int j = 0; j < HID; ++j) z += w[j] * h1[j];
        const float a = tanhf(z);
        h2[i] = a;
        y += sP[OFF_W3 + i] * a;
    }
    return y;
}

__global__ void k_mlp_forward(const float *__restrict__ P, const float *__restrict__ X,
                              float *__restrict__ Y, int n)
{
    extern __shared__ float sP[];
    load_params(P, sP);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float h1[HID], h2[HID];
    Y[s] = mlp_fwd1(sP, X[3 * s], X[3 * s + 1], X[3 * s + 2], h1, h2);
}

// Gradient of the mean squared error over one tile of TILE samples, written to partial[tile], by a
// cluster of two CTAs with SUB samples each; the two add their sums through distributed shared memory,
// each for one half of the parameters.  Every sum has a fixed order, so the result is the same on
// every run.
//
// Bound by float32 FMA (three 64 x 64 x SUB products: layer 2, its transpose for the backward pass, its
// weight gradient; 256 threads with 4 x 4 outputs each, operands in 16-byte loads from rows of ROW
// floats, which meets every bank once) and by the latency of the phases between them.  With 64
// samples a CTA the documented 9716 samples give 152 CTAs, one per SM.  One step (gradient, reduction,
// Adam) on 9716 samples: 105 us with one thread per sample and 128 samples a CTA, 22 us.
constexpr int SUB = 64;
constexpr int ROW = HID + 4;
constexpr int GT = 256; // threads of the gradient kernel
static_assert(TILE == 2 * SUB, "two CTAs a tile");

struct GradMem {
    float W2[HID * ROW];  // W2[i][j]; then dz1[s][j]
    float W2T[HID * ROW]; // W2 transposed
    float H1[SUB * ROW];  // h1[s][j]
    float D2[SUB * ROW];  // h2[s][i], then dz2[s][i]
    float g[(NPARAM + 3) & ~3]; // this CTA's gradient
    float W1[HID * 3], b1[HID], b2[HID], W3[HID];
    float x[SUB * 3], target[SUB], dy[SUB], r2[SUB];
};

// acc[a][b] += sum_k A[ts + 16 a][k] Bm[ti + 16 b][k] over k < 64
__device__ __forceinline__ void product_rows(const float *A, const float *Bm, int ts, int ti, float acc[4][4])
{
#pragma unroll 4
    for (int k = 0; k < HID; k += 4) {
        float4 p[4], q[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) p[a] = *reinterpret_cast<const float4 *>(A + (ts + 16 * a) * ROW + k);
#pragma unroll
        for (int b = 0; b < 4; ++b) q[b] = *reinterpret_cast<const float4 *>(Bm + (ti + 16 * b) * ROW + k);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                acc[a][b] += p[a].x * q[b].x;
                acc[a][b] += p[a].y * q[b].y;
                acc[a][b] += p[a].z * q[b].z;
                acc[a][b] += p[a].w * q[b].w;
            }
    }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GT)
    k_mlp_grad_tile(const float *__restrict__ P, const float *__restrict__ X, const float *__restrict__ T, int n,
                    float *__restrict__ partial, float *__restrict__ loss_partial)
{
    extern __shared__ __align__(16) unsigned char smem[];
    GradMem &M = *reinterpret_cast<GradMem *>(smem);
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int t = threadIdx.x, ti = t & 15, ts = t >> 4;
    const int base = blockIdx.x * SUB, tile = blockIdx.x >> 1;
    float w2[HID * HID / GT]; // all loads in flight at once
#pragma unroll
    for (int k = 0; k < HID * HID / GT; ++k) w2[k] = P[OFF_W2 + t + k * GT];
    if (t < HID * 3) M.W1[t] = P[OFF_W1 + t];
    if (t < HID) {
        M.b1[t] = P[OFF_B1 + t];
        M.b2[t] = P[OFF_B2 + t];
        M.W3[t] = P[OFF_W3 + t];
    }
    if (t < SUB) M.target[t] = base + t < n ? T[base + t] : 0.f;
    if (t < SUB * 3) M.x[t] = base + t / 3 < n ? X[3 * (size_t)base + t] : 0.f;
    const float b3 = P[OFF_B3];
#pragma unroll
    for (int k = 0; k < HID * HID / GT; ++k) {
        const int e = t + k * GT;
        M.W2[(e / HID) * ROW + e % HID] = w2[k];
        M.W2T[(e % HID) * ROW + e / HID] = w2[k];
    }
    __syncthreads();
#pragma unroll 4
    for (int e = t; e < SUB * HID; e += GT) { // layer 1
        const int q = e / HID, j = e % HID;
        const float z = M.b1[j] + M.W1[3 * j] * M.x[3 * q] + M.W1[3 * j + 1] * M.x[3 * q + 1] + M.W1[3 * j + 2] * M.x[3 * q + 2];
        M.H1[q * ROW + j] = tanhf(z);
    }
    __syncthreads();
    float acc[4][4];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) acc[a][b] = M.b2[ti + 16 * b];
    product_rows(M.H1, M.W2, ts, ti, acc); // z2[s][i]
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int q = ts + 16 * a;
        float y = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            acc[a][b] = tanhf(acc[a][b]);
            M.D2[q * ROW + ti + 16 * b] = acc[a][b];
            y += M.W3[ti + 16 * b] * acc[a][b];
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
        y += b3;
        if (ti == 0) {
            const float r = base + q < n ? y - M.target[q] : 0.f;
            M.dy[q] = 2.0f * r / (float)n;
            M.r2[q] = r * r;
        }
    }
    __syncthreads();
    // sums over samples, four threads a unit (16 samples each, then in order)
    const int u = t >> 2, part = t & 3;
    auto over_samples = [&](auto f) {
        float g = 0.f;
#pragma unroll 4
        for (int q = part * (SUB / 4); q < (part + 1) * (SUB / 4); ++q) g += f(q);
        g += __shfl_xor_sync(0xffffffffu, g, 1);
        g += __shfl_xor_sync(0xffffffffu, g, 2);
        return g;
    };
    {
        const float g = over_samples([&](int q) { return M.dy[q] * M.D2[q * ROW + u]; });
        if (part == 0) M.g[OFF_W3 + u] = g;
    }
    float tot = 0.f; // warp 0: db3, warp 1: the loss
    if (t < 64) {
        const float *v = t < 32 ? M.dy : M.r2;
        tot = v[t & 31] + v[(t & 31) + 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        if (t == 0) M.g[OFF_B3] = tot;
    }
    __syncthreads();
    if (t == 32) M.r2[0] = tot; // read by the tile's first CTA below
#pragma unroll
    for (int a = 0; a < 4; ++a) { // dz2 = dy W3 (1 - h2^2)
        const int q = ts + 16 * a;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            M.D2[q * ROW + ti + 16 * b] = M.dy[q] * M.W3[ti + 16 * b] * (1.f - acc[a][b] * acc[a][b]);
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    product_rows(M.D2, M.W2T, ts, ti, acc); // sum_i dz2[s][i] W2[i][j]
#pragma unroll
    for (int a = 0; a < 4; ++a) { // dz1, over W2 (read for the last time before the barriers above)
        const int q = ts + 16 * a;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float h = M.H1[q * ROW + ti + 16 * b];
            M.W2[q * ROW + ti + 16 * b] = acc[a][b] * (1.f - h * h);
        }
    }
    { // dW2[i][j] = sum_s dz2[s][i] h1[s][j], i = 4 ts .., j = 4 ti ..
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
#pragma unroll 4
        for (int q = 0; q < SUB; ++q) {
            const float4 d = *reinterpret_cast<const float4 *>(M.D2 + q * ROW + 4 * ts);
            const float4 h = *reinterpret_cast<const float4 *>(M.H1 + q * ROW + 4 * ti);
            const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += dv[a] * hv[b];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
            *reinterpret_cast<float4 *>(M.g + OFF_W2 + (4 * ts + a) * HID + 4 * ti) =
                make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
    }
    {
        const float g = over_samples([&](int q) { return M.D2[q * ROW + u]; });
        if (part == 0) M.g[OFF_B2 + u] = g;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c) { // W1[j][c] (c < 3) and b1[j] (c == 3)
        const float g = over_samples([&](int q) { return M.W2[q * ROW + u] * (c < 3 ? M.x[3 * q + c] : 1.f); });
        if (part == 0) M.g[c < 3 ? OFF_W1 + 3 * u + c : OFF_B1 + u] = g;
    }
    cluster.sync();
    const unsigned rank = cluster.block_rank();
    const GradMem &O = *cluster.map_shared_rank(&M, rank ^ 1u);
    float *out = partial + (size_t)tile * NPARAM;
    float other[NPARAM / 2 / GT + 1]; // all loads in flight at once
#pragma unroll
    for (int k = 0; k < NPARAM / 2 / GT + 1; ++k) {
        const int p = t + k * GT + (rank ? NPARAM / 2 : 0);
        other[k] = p < (rank ? NPARAM : NPARAM / 2) ? O.g[p] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < NPARAM / 2 / GT + 1; ++k) {
        const int p = t + k * GT + (rank ? NPARAM / 2 : 0);
        if (p < (rank ? NPARAM : NPARAM / 2)) out[p] = rank ? other[k] + M.g[p] : M.g[p] + other[k];
    }
    if (rank == 0 && t == 0) loss_partial[tile] = M.r2[0] + O.r2[0];
    cluster.sync(); // the other CTA has read this one's sums
}

// One Adam step (Kingma & Ba 2015), bias-corrected, step t >= 1, of one parameter
__device__ __forceinline__ void adam_step(float *P, float *m, float *v, float gp, int t, float lr, float b1, float b2,
                                          float eps)
{
    const float mp = b1 * *m + (1.f - b1) * gp;
    const float vp = b2 * *v + (1.f - b2) * gp * gp;
    *m = mp;
    *v = vp;
    const float mh = mp / (1.f - powf(b1, (float)t));
    const float vh = vp / (1.f - powf(b2, (float)t));
    *P -= lr * mh / (sqrtf(vh) + eps);
}

// grad[p] = sum over tiles of partial[tile][p]: eight threads a parameter take every eighth tile each,
// then their sums are added in order; loss = sum of tile losses / n.  step >= 1: that Adam step too.
constexpr int RED_P = 32, RED_S = 8;

__global__ void __launch_bounds__(RED_P *RED_S)
    k_mlp_reduce(const float *__restrict__ partial, const float *__restrict__ lpart, int ntiles, int n,
                 float *__restrict__ grad, float *__restrict__ loss, float *__restrict__ P, float *__restrict__ m,
                 float *__restrict__ v, int step, float lr, float b1, float b2, float eps)
{
    __shared__ float sums[RED_S][RED_P + 1];
    const int i = threadIdx.x % RED_P, q = threadIdx.x / RED_P, p = blockIdx.x * RED_P + i;
    float g = 0.f;
    if (p < NPARAM)
#pragma unroll 10
        for (int k = q; k < ntiles; k += RED_S) g += partial[(size_t)k * NPARAM + p];
    sums[q][i] = g;
    __syncthreads();
    if (q == 0 && p < NPARAM) {
        g = 0.f;
#pragma unroll
        for (int k = 0; k < RED_S; ++k) g += sums[k][i];
        grad[p] = g;
        if (step > 0) adam_step(P + p, m + p, v + p, g, step, lr, b1, b2, eps);
    }
    if (blockIdx.x == 0 && q == 1 && loss) { // one warp
        float l = 0.f;
        for (int k = i; k < ntiles; k += 32) l += lpart[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (i == 0) *loss = l / (float)n;
    }
}

__global__ void k_mlp_adam(float *__restrict__ P, const float *__restrict__ g, float *__restrict__ m,
                           float *__restrict__ v, int t, float lr, float b1, float b2, float eps)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < NPARAM) adam_step(P + p, m + p, v + p, g[p], t, lr, b1, b2, eps);
}

// Glorot-uniform weights from Philox (key = seed), zero biases.
__global__ void k_mlp_init(float *__restrict__ P, uint32_t k0, uint32_t k1)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NPARAM) return;
    const rewl::u32x4 r = rewl::philox((uint32_t)p, 0u, 0u, 0x4d4c5000u, k0, k1);
    const float u = ((float)(r.x >> 8) + 0.5f) * 0x1p-24f * 2.f - 1.f; // (-1, 1)
    float a = 0.f;
    if (p < OFF_B1) a = sqrtf(6.f / (3 + HID));
    else if (p >= OFF_W2 && p < OFF_B2) a = sqrtf(6.f / (HID + HID));
    else if (p >= OFF_W3 && p < OFF_B3) a = sqrtf(6.f / (HID + 1));
    P[p] = a * u;
}

// Features and targets of a converged ln g: one sample per reachable bin, in bin order (one
// CTA of 1024 threads, block-wide scans), so the training sums always see the same order.
__global__ void __launch_bounds__(1024) k_mlp_samples(const double *__restrict__ lng, int B, int model,
                                                      int q, int L, float *__restrict__ X,
                                                      float *__restrict__ T, int *__restrict__ count)
{
    __shared__ int wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int N = L * L;
    int base = 0;
    for (int b0 = 0; b0 <= B; b0 += blockDim.x) {
        const int b = b0 + threadIdx.x;
        const double v = b <= B ? lng[b] : -INFINITY;
        const int f = v > -INFINITY ? 1 : 0;
        int x = f; // inclusive warp scan
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        if (wid == 0) {
            int w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            wsum[lane] = w; // inclusive prefix over warps
        }
        __syncthreads();
        const int pos = base + (wid ? wsum[wid - 1] : 0) + x - f;
        if (f) {
            const double e = model == 0 ? -2.0 + 2.0 * (double)b / N : -2.0 + (double)b / N;
            X[3 * pos] = (float)e;
            X[3 * pos + 1] = (float)q;
            X[3 * pos + 2] = 1.0f / (float)L;
            T[pos] = (float)(v / N);
        }
        base += wsum[(blockDim.x >> 5) - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = base;
}

// ln g(E) = N * net(e, q, 1/L) for every bin of the target lattice (float64 output).
__global__ void k_mlp_predict(const float *__restrict__ P, int B, int model, int q, int L,
                              double *__restrict__ out)
{
    extern __shared__ float sP[];
    load_params(P, sP);
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > B) return;
    const int N = L * L;
    const float e = model == 0 ? -2.0f + 2.0f * (float)b / N : -2.0f + (float)b / N;
    float h1[HID], h2[HID];
    out[b] = (double)N * (double)mlp_fwd1(sP, e, (float)q, 1.0f / (float)L, h1, h2);
}

int fail(cudaError_t e, const char *where)
{
    g_mlp_err = std::string(where) + ": " + cudaGetErrorString(e);
    return REWL_ERR_CUDA;
}

} // namespace

extern "C" {

int rewl_mlp_forward(const float *P, const float *X, float *Y, int n, void *stream)
{
    if (!P || !X || !Y || n < 0) return REWL_ERR_INVALID_ARG;
    if (n == 0) return REWL_OK;
    k_mlp_forward<<<(n + 127) / 128, 128, NPARAM * sizeof(float), (cudaStream_t)stream>>>(P, X, Y, n);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REWL_OK : fail(e, "rewl_mlp_forward");
}

int rewl_mlp_workspace_floats(int n) { return ((n + TILE - 1) / TILE) * (NPARAM + 1) + 1; }

// gradient and, with step >= 1, that Adam step, in two launches
static int grad_and_step(float *P, const float *X, const float *T, int n, float *grad, float *loss, float *work,
                         float *m, float *v, int step, double lr, cudaStream_t st)
{
    const int ntiles = (n + TILE - 1) / TILE;
    float *partial = work, *lpart = work + (size_t)ntiles * NPARAM;
    k_mlp_grad_tile<<<2 * ntiles, GT, sizeof(GradMem), st>>>(P, X, T, n, partial, lpart);
    k_mlp_reduce<<<(NPARAM + RED_P - 1) / RED_P, RED_P * RED_S, 0, st>>>(partial, lpart, ntiles, n, grad, loss, P, m, v,
                                                                       step, (float)lr, 0.9f, 0.999f, 1e-8f);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REWL_OK : fail(e, "rewl_mlp_grad");
}

static cudaError_t grad_ready()
{
    return cudaFuncSetAttribute(k_mlp_grad_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradMem));
}

int rewl_mlp_grad(const float *P, const float *X, const float *T, int n, float *grad, float *loss,
                  float *work, void *stream)
{
    if (!P || !X || !T || !grad || !work || n < 1) return REWL_ERR_INVALID_ARG;
    const cudaError_t e = grad_ready();
    if (e != cudaSuccess) return fail(e, "rewl_mlp_grad");
    return grad_and_step(const_cast<float *>(P), X, T, n, grad, loss, work, nullptr, nullptr, 0, 0.0, (cudaStream_t)stream);
}

int rewl_mlp_adam(float *P, const float *grad, float *m, float *v, int t, double lr, void *stream)
{
    if (!P || !grad || !m || !v || t < 1 || !(lr > 0)) return REWL_ERR_INVALID_ARG;
    k_mlp_adam<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(P, grad, m, v, t, (float)lr,
                                                                       0.9f, 0.999f, 1e-8f);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REWL_OK : fail(e, "rewl_mlp_adam");
}

int rewl_mlp_train(float *P, const float *X, const float *T, int n, int steps, double lr,
                   int t0, float *m, float *v, float *grad, float *work, float *loss_out,
                   void *stream)
{
    if (!P || !X || !T || !m || !v || !grad || !work || n < 1 || steps < 0 || t0 < 0)
        return REWL_ERR_INVALID_ARG;
    const cudaError_t e = grad_ready();
    if (e != cudaSuccess) return fail(e, "rewl_mlp_train");
    for (int s = 0; s < steps; ++s) {
        float *loss = s + 1 == steps ? loss_out : nullptr;
        const int rc = grad_and_step(P, X, T, n, grad, loss, work, m, v, lr > 0 ? t0 + s + 1 : 0, lr, (cudaStream_t)stream);
        if (rc != REWL_OK) return rc;
        if (!(lr > 0)) return REWL_ERR_INVALID_ARG;
    }
    return REWL_OK;
}

int rewl_mlp_init(float *P, uint64_t seed, void *stream)
{
    if (!P) return REWL_ERR_INVALID_ARG;
    k_mlp_init<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(P, (uint32_t)seed,
                                                                       (uint32_t)(seed >> 32));
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REWL_OK : fail(e, "rewl_mlp_init");
}

int rewl_mlp_samples(const double *lng, int model, int L, float *X, float *T, int *count,
                     void *stream)
{
    if (!lng || !X || !T || !count || L < 2 || (model != 0 && model < 2)) return REWL_ERR_INVALID_ARG;
    const int N = L * L, B = model == 0 ? N : 2 * N, q = model == 0 ? 2 : model;
    k_mlp_samples<<<1, 1024, 0, (cudaStream_t)stream>>>(lng, B, model, q, L, X, T, count);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REWL_OK : fail(e, "rewl_mlp_samples");
}

int rewl_mlp_predict(const float *P, int model, int L, double *lng, void *stream)
{
    if (!P || !lng || L < 2 || (model != 0 && model < 2)) return REWL_ERR_INVALID_ARG;
    const int N = L * L, B = model == 0 ? N : 2 * N, q = model == 0 ? 2 : model;
    k_mlp_predict<<<(B + 128) / 128, 128, NPARAM * sizeof(float), (cudaStream_t)stream>>>(P, B, model,
                                                                                        q, L, lng);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? REWL_OK : fail(e, "rewl_mlp_predict");
}

const char *rewl_mlp_last_error(void) { return g_mlp_err.c_str(); }

} // extern "C"
