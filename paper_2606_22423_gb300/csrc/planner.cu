// Learned planner: a small FP32 network (4 -> 64 -> 64 -> S, ReLU) that
// predicts the log time of each scan strategy for a column from four
// features, trained on the GPU by these kernels (forward, backward, Adam).
// Every scan strategy returns the same exact result, so the planner only
// affects speed.
//
// Layout: parameters are one flat float array [W1 (4x64), b1, W2 (64x64), b2,
// W3 (64xS), b3], W_l row-major with shape (fan_in, fan_out).  Gradients are summed
// per CTA over its rows and then over the CTAs in a fixed order (no atomics, so a
// training step is deterministic).
//
// Bound: latency -- 19 KB of weights and a few thousand multiply-adds per row.  The
// whole network is one kernel over tiles of 16 rows with weights and activations in
// shared memory, and a gradient one more that adds the CTAs' partial sums (and takes
// the Adam step).  One kernel per layer and direction, ten launches with weight
// gradients summed over all rows by one thread each, took 111 us for a forward pass of
// 4096 rows and a gradient of 160.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/gbscan.h"
#include "batch_kernels.cuh"
#include "internal.h"

namespace {

constexpr int kIn = 4;
constexpr int kHid = 64;
constexpr uint32_t kCkptMagic = 0x4e4c5047u;  // "GPLN"
constexpr uint32_t kCkptVersion = 1;

scan_status pfail(scan_status s, const char* msg)
{
    gb_set_last_error(msg);
    return s;
}

scan_status pcuda(cudaError_t e, const char* what)
{
    static thread_local char buf[256];
    snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    gb_set_last_error(buf);
    return gb_cuda_status(e);
}

#define PL_CUDA(call)                                  \
    do {                                               \
        cudaError_t e_ = (call);                       \
        if (e_ != cudaSuccess) return pcuda(e_, #call); \
    } while (0)

constexpr int kTileRows = 16;
constexpr int kThreads = 256;          // 64 units x 4 groups of 4 rows
constexpr int kMaxOut = 16;            // strategies
constexpr int kPadW2 = kHid + 1;       // W2's rows are read along both axes
constexpr int kMaxParts = 48;          // CTAs of a gradient pass, each with its partial sums (0.9 MB in all)

__host__ __device__ constexpr int param_count(int S) { return kIn * kHid + kHid + kHid * kHid + kHid + kHid * S + S; }

struct Net {  // the parameters in shared memory
    float W1[kIn * kHid], b1[kHid], W2[kHid * kPadW2], b2[kHid], W3[kHid * kMaxOut], b3[kMaxOut];
};

struct Tile {  // activations and their gradients of one tile
    float x[kTileRows][kIn];
    float a1[kTileRows][kHid + 4], a2[kTileRows][kHid + 1];
    float dy[kTileRows][kMaxOut], dz2[kTileRows][kHid], dz1[kTileRows][kHid];
};

__device__ void load_net(Net& n, const float* __restrict__ P, int S)
{
    const int t = threadIdx.x;
    for (int i = t; i < kIn * kHid + kHid; i += kThreads) (i < kIn * kHid ? n.W1[i] : n.b1[i - kIn * kHid]) = P[i];
    P += kIn * kHid + kHid;
#pragma unroll
    for (int i = t; i < kHid * kHid; i += kThreads) n.W2[(i >> 6) * kPadW2 + (i & 63)] = P[i];
    P += kHid * kHid;
    if (t < kHid) n.b2[t] = P[t];
    P += kHid;
    for (int i = t; i < kHid * S + S; i += kThreads) (i < kHid * S ? n.W3[i] : n.b3[i - kHid * S]) = P[i];
}

// Rows row0 .. row0 + 15: x, a1 and a2 into the tile (zero inputs past `rows`).
__device__ void forward_tile(const Net& n, Tile& T, const float* __restrict__ x, int row0, int rows)
{
    const int t = threadIdx.x, m = t & 63, r0 = (t >> 6) * 4;
    if (t < kTileRows * kIn) T.x[t / kIn][t % kIn] = row0 + t / kIn < rows ? x[row0 * kIn + t] : 0.f;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float acc = n.b1[m];
#pragma unroll
        for (int k = 0; k < kIn; ++k) acc = fmaf(T.x[r0 + r][k], n.W1[k * kHid + m], acc);
        T.a1[r0 + r][m] = acc > 0.f ? acc : 0.f;
    }
    __syncthreads();
    float acc[4] = {n.b2[m], n.b2[m], n.b2[m], n.b2[m]};
#pragma unroll
    for (int k = 0; k < kHid; k += 4) {
        float w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = n.W2[(k + j) * kPadW2 + m];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float4 a = *reinterpret_cast<const float4*>(&T.a1[r0 + r][k]);
            acc[r] = fmaf(a.x, w[0], acc[r]);
            acc[r] = fmaf(a.y, w[1], acc[r]);
            acc[r] = fmaf(a.z, w[2], acc[r]);
            acc[r] = fmaf(a.w, w[3], acc[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) T.a2[r0 + r][m] = acc[r] > 0.f ? acc[r] : 0.f;
    __syncthreads();
}

__device__ float output(const Net& n, const Tile& T, int r, int s, int S)
{
    float acc = n.b3[s];
#pragma unroll 16
    for (int k = 0; k < kHid; ++k) acc = fmaf(T.a2[r][k], n.W3[k * S + s], acc);
    return acc;
}

__global__ void __launch_bounds__(kThreads) k_forward(const float* __restrict__ P, int S, const float* __restrict__ x,
                                                      int rows, float* __restrict__ y)
{
    __shared__ Net n;
    __shared__ __align__(16) Tile T;
    load_net(n, P, S);
    for (int row0 = static_cast<int>(blockIdx.x) * kTileRows; row0 < rows;
         row0 += static_cast<int>(gridDim.x) * kTileRows) {
        __syncthreads();
        forward_tile(n, T, x, row0, rows);
        const int r = static_cast<int>(threadIdx.x) / S, s = static_cast<int>(threadIdx.x) % S;
        if (r < kTileRows && row0 + r < rows) y[(row0 + r) * S + s] = output(n, T, r, s, S);
    }
}

// Partial gradients of mean((y - t)^2) over this CTA's rows, and its part of the loss
// after them: part[blockIdx.x][param_count(S) + 1].  A ReLU's z > 0 is its a > 0.
__global__ void __launch_bounds__(kThreads) k_gradients(const float* __restrict__ P, int S,
                                                        const float* __restrict__ x, const float* __restrict__ t,
                                                        int rows, float* __restrict__ part)
{
    __shared__ Net n;
    __shared__ __align__(16) Tile T;
    __shared__ float red[kThreads / 32];
    const int tid = threadIdx.x, m = tid & 63, q = tid >> 6;
    load_net(n, P, S);
    float g1 = 0.f, gb1 = 0.f, gb2 = 0.f, g2[16] = {}, g3[4] = {}, gb3 = 0.f, loss = 0.f;
    const float count = static_cast<float>(rows * S);
    for (int row0 = static_cast<int>(blockIdx.x) * kTileRows; row0 < rows;
         row0 += static_cast<int>(gridDim.x) * kTileRows) {
        __syncthreads();
        forward_tile(n, T, x, row0, rows);
        const int ro = tid / S, so = tid % S;
        if (ro < kTileRows) {
            float dy = 0.f;
            if (row0 + ro < rows) {
                const float d = output(n, T, ro, so, S) - t[(row0 + ro) * S + so];
                dy = 2.f * d / count;
                loss += d * d / count;
            }
            T.dy[ro][so] = dy;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float acc = 0.f;
            for (int s = 0; s < S; ++s) acc = fmaf(T.dy[4 * q + r][s], n.W3[m * S + s], acc);
            T.dz2[4 * q + r][m] = T.a2[4 * q + r][m] > 0.f ? acc : 0.f;
        }
        __syncthreads();
        float acc[4] = {};
#pragma unroll 16
        for (int j = 0; j < kHid; ++j) {
            const float w = n.W2[m * kPadW2 + j];
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] = fmaf(T.dz2[4 * q + r][j], w, acc[r]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) T.dz1[4 * q + r][m] = T.a1[4 * q + r][m] > 0.f ? acc[r] : 0.f;
        __syncthreads();
        // this thread's weights: W2[16q .. 16q + 15][m], W1[q][m], a bias, every 256th of W3
#pragma unroll
        for (int r = 0; r < kTileRows; ++r) {
            const float d2 = T.dz2[r][m], d1 = T.dz1[r][m];
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
                const float4 a = *reinterpret_cast<const float4*>(&T.a1[r][16 * q + k]);
                g2[k] = fmaf(a.x, d2, g2[k]);
                g2[k + 1] = fmaf(a.y, d2, g2[k + 1]);
                g2[k + 2] = fmaf(a.z, d2, g2[k + 2]);
                g2[k + 3] = fmaf(a.w, d2, g2[k + 3]);
            }
            g1 = fmaf(T.x[r][q], d1, g1);
            gb1 += d1;
            gb2 += d2;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i = tid + e * kThreads;
            if (i < kHid * S)
                for (int r = 0; r < kTileRows; ++r) g3[e] = fmaf(T.a2[r][i / S], T.dy[r][i % S], g3[e]);
        }
        if (tid < S)
            for (int r = 0; r < kTileRows; ++r) gb3 += T.dy[r][tid];
    }
    float* G = part + static_cast<size_t>(blockIdx.x) * (param_count(S) + 1);
    G[q * kHid + m] = g1;
    if (q == 0) G[kIn * kHid + m] = gb1;
    float* G2 = G + kIn * kHid + kHid;
#pragma unroll
    for (int k = 0; k < 16; ++k) G2[(16 * q + k) * kHid + m] = g2[k];
    if (q == 1) G2[kHid * kHid + m] = gb2;
    float* G3 = G2 + kHid * kHid + kHid;
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (tid + e * kThreads < kHid * S) G3[tid + e * kThreads] = g3[e];
    if (tid < S) G3[kHid * S + tid] = gb3;
#pragma unroll
    for (int o = 16; o; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if ((tid & 31) == 0) red[tid >> 5] = loss;
    __syncthreads();
    if (tid == 0) {
        float l = 0.f;
        for (int w = 0; w < kThreads / 32; ++w) l += red[w];
        G[param_count(S)] = l;
    }
}

struct Adam {
    int on;
    float lr, b1, b2, eps, bc1, bc2;
};

// Adds the parts in CTA order: gradients to g (and out, if given), the loss after
// them, and one Adam step where asked.
__global__ void __launch_bounds__(128) k_reduce(const float* __restrict__ part, int parts, int count,
                                                float* __restrict__ g, float* __restrict__ out,
                                                float* __restrict__ loss, Adam ad, float* __restrict__ p,
                                                float* __restrict__ m, float* __restrict__ v)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > count) return;
    float gi = 0.f;
#pragma unroll 8
    for (int c = 0; c < parts; ++c) gi += part[static_cast<size_t>(c) * (count + 1) + i];
    if (i == count) {
        *loss = gi;
        return;
    }
    g[i] = gi;
    if (out) out[i] = gi;
    if (!ad.on) return;
    const float mi = ad.b1 * m[i] + (1.f - ad.b1) * gi;
    const float vi = ad.b2 * v[i] + (1.f - ad.b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= ad.lr * (mi / ad.bc1) / (sqrtf(vi / ad.bc2) + ad.eps);
}

// The first strategy (in index order) whose predicted log time is within
// `margin` of the row's minimum: with margin 0 the argmin (ties to the lower
// index); with margin > 0 predicted gains below the margin do not move the
// plan off the earlier (simpler) strategies.
__global__ void k_argmin_rows(const float* __restrict__ y, int rows, int S, float margin,
                              int32_t* __restrict__ out)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= rows) return;
    float lo = y[n * S];
    for (int s = 1; s < S; ++s) lo = fminf(lo, y[n * S + s]);
    int best = 0;
    while (best < S - 1 && y[n * S + best] > lo + margin) ++best;
    out[n] = best;
}

// Same rule on y + prior: the network predicts a correction to a prior
// estimate of each strategy's log time (the law's), row-major rows x S.
__global__ void k_argmin_rows_prior(const float* __restrict__ y, const float* __restrict__ prior, int rows,
                                    int S, float margin, int32_t* __restrict__ out)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= rows) return;
    float lo = y[n * S] + prior[n * S];
    for (int s = 1; s < S; ++s) lo = fminf(lo, y[n * S + s] + prior[n * S + s]);
    int best = 0;
    while (best < S - 1 && y[n * S + best] + prior[n * S + best] > lo + margin) ++best;
    out[n] = best;
}

// Bounds of the features the network was trained on: outside them its
// predictions are extrapolations, and the fallback decides.
struct FeatureBox {
    float lo[kIn], hi[kIn];
    int on;
};

// The fallback's choice unless the network is confident and on familiar
// ground: per row whose features lie inside the box, the strategy the network
// predicts fastest among those available (the fallback's log time below
// kUnavailable) replaces the fallback's choice only if its predicted log time
// is lower than the network's prediction for the fallback's choice by more
// than `margin`.
constexpr float kUnavailable = 29.0f;
__global__ void k_choose_guarded(const float* __restrict__ x, const float* __restrict__ y,
                                 const int32_t* __restrict__ fallback, const float* __restrict__ fallback_log_ms,
                                 int rows, int S, float margin, FeatureBox box, int32_t* __restrict__ out)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= rows) return;
    const int f = fallback[n];
    if (box.on) {
        for (int k = 0; k < kIn; ++k) {
            const float v = x[n * kIn + k];
            if (v < box.lo[k] || v > box.hi[k]) {
                out[n] = f;
                return;
            }
        }
    }
    int best = f;
    for (int s = 0; s < S; ++s) {
        if (fallback_log_ms[n * S + s] >= kUnavailable) continue;
        if (y[n * S + s] < y[n * S + best]) best = s;
    }
    out[n] = (y[n * S + best] < y[n * S + f] - margin) ? best : f;
}

inline unsigned blocks_for(long long n, int t = 256) { return static_cast<unsigned>((n + t - 1) / t); }

// splitmix64 (Steele, Lea, Flood 2014) for the deterministic initial weights
uint64_t splitmix64(uint64_t& s)
{
    uint64_t z = (s += 0x9e3779b97f4a7c15ull);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

}  // namespace

struct scan_planner {
    int S = 4;
    size_t nparams = 0;
    float* d_params = nullptr;
    float* d_grads = nullptr;
    float* d_m = nullptr;
    float* d_v = nullptr;
    int step = 0;
    int cap = 0;  // rows of the output workspace (the choices' predictions)
    float* d_ws = nullptr;
    float* d_part = nullptr;  // partial gradients, kMaxParts of them
    float* d_loss = nullptr;

    size_t off_W(int l) const
    {
        const int fi[3] = {kIn, kHid, kHid}, fo[3] = {kHid, kHid, S};
        size_t o = 0;
        for (int i = 0; i < l; ++i) o += static_cast<size_t>(fi[i]) * fo[i] + fo[i];
        return o;
    }
    size_t off_b(int l) const
    {
        const int fi[3] = {kIn, kHid, kHid}, fo[3] = {kHid, kHid, S};
        return off_W(l) + static_cast<size_t>(fi[l]) * fo[l];
    }
};

namespace {

scan_status ensure_ws(scan_planner* pl, uint32_t rows)
{
    if (static_cast<int>(rows) <= pl->cap) return SCAN_OK;
    if (pl->d_ws) cudaFree(pl->d_ws);
    pl->d_ws = nullptr;
    PL_CUDA(cudaMalloc(&pl->d_ws, static_cast<size_t>(pl->S) * rows * sizeof(float)));
    pl->cap = static_cast<int>(rows);
    return SCAN_OK;
}

void forward(const scan_planner* pl, const float* x, int rows, float* y, cudaStream_t st)
{
    const unsigned tiles = static_cast<unsigned>((rows + kTileRows - 1) / kTileRows);
    k_forward<<<std::min(tiles, 1024u), kThreads, 0, st>>>(pl->d_params, pl->S, x, rows, y);
}

// Gradients (and, with ad.on, the Adam step) on st; the loss goes to d_loss.
scan_status gradients(scan_planner* pl, const float* x, const float* t, uint32_t rows, float* out, const Adam& ad,
                      cudaStream_t st)
{
    const int count = static_cast<int>(pl->nparams);
    const int tiles = static_cast<int>((rows + kTileRows - 1) / kTileRows);
    const int parts = std::min(tiles, kMaxParts);
    k_gradients<<<parts, kThreads, 0, st>>>(pl->d_params, pl->S, x, t, static_cast<int>(rows), pl->d_part);
    k_reduce<<<blocks_for(count + 1, 128), 128, 0, st>>>(pl->d_part, parts, count, pl->d_grads, out, pl->d_loss, ad,
                                                         pl->d_params, pl->d_m, pl->d_v);
    PL_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status read_loss(scan_planner* pl, cudaStream_t st, float* host_loss)
{
    if (!host_loss) return SCAN_OK;
    PL_CUDA(cudaMemcpyAsync(host_loss, pl->d_loss, sizeof(float), cudaMemcpyDeviceToHost, st));
    PL_CUDA(cudaStreamSynchronize(st));
    return SCAN_OK;
}

}  // namespace

extern "C" {

scan_status scan_planner_create(uint32_t n_strategies, uint64_t seed, scan_planner** out)
{
    gb_set_last_error("");
    if (!out || n_strategies < 1 || n_strategies > 16) return pfail(SCAN_EINVAL, "bad planner shape");
    auto* pl = new (std::nothrow) scan_planner();
    if (!pl) return pfail(SCAN_ENOMEM, "host allocation failed");
    pl->S = static_cast<int>(n_strategies);
    pl->nparams = pl->off_b(2) + pl->S;
    std::vector<float> h(pl->nparams, 0.f);
    uint64_t s = seed;
    const int fi[3] = {kIn, kHid, kHid}, fo[3] = {kHid, kHid, pl->S};
    for (int l = 0; l < 3; ++l) {  // He-uniform weights, zero biases
        const float lim = std::sqrt(6.f / static_cast<float>(fi[l]));
        for (int i = 0; i < fi[l] * fo[l]; ++i) {
            const double u = static_cast<double>(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0);
            h[pl->off_W(l) + i] = static_cast<float>((2.0 * u - 1.0) * lim);
        }
    }
    // parameters, gradients, Adam's moments, the loss; then a gradient pass's partial sums
    cudaError_t e = cudaMalloc(&pl->d_params, (4 * pl->nparams + 4 + kMaxParts * (pl->nparams + 1)) * sizeof(float));
    if (e != cudaSuccess) {
        delete pl;
        return pcuda(e, "cudaMalloc(planner)");
    }
    pl->d_grads = pl->d_params + pl->nparams;
    pl->d_m = pl->d_grads + pl->nparams;
    pl->d_v = pl->d_m + pl->nparams;
    pl->d_loss = pl->d_v + pl->nparams;
    pl->d_part = pl->d_loss + 4;
    e = cudaMemset(pl->d_params, 0, 4 * pl->nparams * sizeof(float) + 16);
    if (e == cudaSuccess) e = cudaMemcpy(pl->d_params, h.data(), pl->nparams * sizeof(float), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(pl->d_params);
        delete pl;
        return pcuda(e, "planner init");
    }
    *out = pl;
    return SCAN_OK;
}

scan_status scan_planner_destroy(scan_planner* pl)
{
    if (!pl) return SCAN_OK;
    cudaDeviceSynchronize();
    if (pl->d_params) cudaFree(pl->d_params);
    if (pl->d_ws) cudaFree(pl->d_ws);
    delete pl;
    return SCAN_OK;
}

uint64_t scan_planner_param_count(const scan_planner* pl) { return pl ? pl->nparams : 0; }

scan_status scan_planner_get_params(const scan_planner* pl, float* host_params)
{
    if (!pl || !host_params) return pfail(SCAN_EINVAL, "null pointer");
    PL_CUDA(cudaMemcpy(host_params, pl->d_params, pl->nparams * sizeof(float), cudaMemcpyDeviceToHost));
    return SCAN_OK;
}

scan_status scan_planner_set_params(scan_planner* pl, const float* host_params)
{
    if (!pl || !host_params) return pfail(SCAN_EINVAL, "null pointer");
    PL_CUDA(cudaMemcpy(pl->d_params, host_params, pl->nparams * sizeof(float), cudaMemcpyHostToDevice));
    PL_CUDA(cudaMemset(pl->d_m, 0, 2 * pl->nparams * sizeof(float)));
    pl->step = 0;
    return SCAN_OK;
}

scan_status scan_planner_forward(scan_planner* pl, const float* dev_x, uint32_t rows, float* dev_y, void* stream)
{
    gb_set_last_error("");
    if (!pl || (rows && (!dev_x || !dev_y))) return pfail(SCAN_EINVAL, "null pointer");
    if (!rows) return SCAN_OK;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t x_bytes = sizeof(float) * kIn * rows, y_bytes = sizeof(float) * static_cast<size_t>(pl->S) * rows;
    const uintptr_t x0 = reinterpret_cast<uintptr_t>(dev_x), y0 = reinterpret_cast<uintptr_t>(dev_y);
    // a tile's predictions are written while other tiles' features are still to be read: a
    // dev_y that shares memory with dev_x gets them after the kernel
    const bool shared = x0 < y0 + y_bytes && y0 < x0 + x_bytes;
    float* y = dev_y;
    if (shared) {
        const scan_status s = ensure_ws(pl, rows);
        if (s != SCAN_OK) return s;
        y = pl->d_ws;
    }
    forward(pl, dev_x, static_cast<int>(rows), y, st);
    PL_CUDA(cudaGetLastError());
    if (shared) PL_CUDA(cudaMemcpyAsync(dev_y, y, y_bytes, cudaMemcpyDeviceToDevice, st));
    return SCAN_OK;
}

scan_status scan_planner_gradients(scan_planner* pl, const float* dev_x, const float* dev_t, uint32_t rows,
                                   float* dev_grads, void* stream, float* host_loss)
{
    gb_set_last_error("");
    if (!pl || !rows || !dev_x || !dev_t) return pfail(SCAN_EINVAL, "null pointer or empty batch");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const scan_status s = gradients(pl, dev_x, dev_t, rows, dev_grads, Adam{}, st);
    if (s != SCAN_OK) return s;
    return read_loss(pl, st, host_loss);
}

scan_status scan_planner_train_step(scan_planner* pl, const float* dev_x, const float* dev_t, uint32_t rows,
                                    float lr, void* stream, float* host_loss)
{
    gb_set_last_error("");
    if (!pl || !rows || !dev_x || !dev_t) return pfail(SCAN_EINVAL, "null pointer or empty batch");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int step = pl->step + 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const Adam ad{1, lr, b1, b2, 1e-8f, 1.f - std::pow(b1, static_cast<float>(step)),
                  1.f - std::pow(b2, static_cast<float>(step))};
    const scan_status s = gradients(pl, dev_x, dev_t, rows, nullptr, ad, st);
    if (s != SCAN_OK) return s;
    pl->step = step;
    return read_loss(pl, st, host_loss);
}

scan_status scan_planner_choose_margin(scan_planner* pl, const float* dev_x, uint32_t rows, float margin,
                                       int32_t* dev_choice, void* stream)
{
    if (!(margin >= 0.0f)) return pfail(SCAN_EINVAL, "margin must be >= 0");
    scan_status s = ensure_ws(pl, rows ? rows : 1);
    if (s != SCAN_OK) return s;
    s = scan_planner_forward(pl, dev_x, rows, pl->d_ws, stream);
    if (s != SCAN_OK || !rows) return s;
    k_argmin_rows<<<blocks_for(rows), 256, 0, static_cast<cudaStream_t>(stream)>>>(pl->d_ws, static_cast<int>(rows),
                                                                                  pl->S, margin, dev_choice);
    PL_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status scan_planner_choose_prior(scan_planner* pl, const float* dev_x, uint32_t rows, float margin,
                                      const float* dev_prior, int32_t* dev_choice, void* stream)
{
    if (!pl || (rows && (!dev_x || !dev_prior || !dev_choice))) return pfail(SCAN_EINVAL, "null pointer");
    if (!(margin >= 0.0f)) return pfail(SCAN_EINVAL, "margin must be >= 0");
    scan_status s = ensure_ws(pl, rows ? rows : 1);
    if (s != SCAN_OK) return s;
    s = scan_planner_forward(pl, dev_x, rows, pl->d_ws, stream);
    if (s != SCAN_OK || !rows) return s;
    k_argmin_rows_prior<<<blocks_for(rows), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        pl->d_ws, dev_prior, static_cast<int>(rows), pl->S, margin, dev_choice);
    PL_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status scan_planner_choose_guarded(scan_planner* pl, const float* dev_x, uint32_t rows, float margin,
                                        const int32_t* dev_fallback, const float* dev_fallback_log_ms,
                                        const float* host_feature_box, int32_t* dev_choice, void* stream)
{
    if (!pl || (rows && (!dev_x || !dev_fallback || !dev_fallback_log_ms || !dev_choice)))
        return pfail(SCAN_EINVAL, "null pointer");
    if (!(margin >= 0.0f)) return pfail(SCAN_EINVAL, "margin must be >= 0");
    scan_status s = ensure_ws(pl, rows ? rows : 1);
    if (s != SCAN_OK) return s;
    s = scan_planner_forward(pl, dev_x, rows, pl->d_ws, stream);
    if (s != SCAN_OK || !rows) return s;
    FeatureBox box{};
    box.on = host_feature_box != nullptr;
    for (int k = 0; k < kIn && box.on; ++k) {
        box.lo[k] = host_feature_box[k];
        box.hi[k] = host_feature_box[kIn + k];
    }
    k_choose_guarded<<<blocks_for(rows), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        dev_x, pl->d_ws, dev_fallback, dev_fallback_log_ms, static_cast<int>(rows), pl->S, margin, box, dev_choice);
    PL_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status scan_planner_choose(scan_planner* pl, const float* dev_x, uint32_t rows, int32_t* dev_choice,
                                void* stream)
{
    return scan_planner_choose_margin(pl, dev_x, rows, 0.0f, dev_choice, stream);
}

scan_status scan_planner_save(const scan_planner* pl, const char* path)
{
    if (!pl || !path) return pfail(SCAN_EINVAL, "null pointer");
    std::vector<float> h(pl->nparams);
    scan_status s = scan_planner_get_params(pl, h.data());
    if (s != SCAN_OK) return s;
    FILE* f = std::fopen(path, "wb");
    if (!f) return pfail(SCAN_EINVAL, "cannot open checkpoint for writing");
    const uint32_t hdr[4] = {kCkptMagic, kCkptVersion, static_cast<uint32_t>(pl->S),
                             static_cast<uint32_t>(pl->nparams)};
    const bool ok = std::fwrite(hdr, sizeof hdr, 1, f) == 1 &&
                    std::fwrite(h.data(), sizeof(float), h.size(), f) == h.size();
    std::fclose(f);
    return ok ? SCAN_OK : pfail(SCAN_EINVAL, "short write of checkpoint");
}

scan_status scan_planner_load(scan_planner* pl, const char* path)
{
    if (!pl || !path) return pfail(SCAN_EINVAL, "null pointer");
    FILE* f = std::fopen(path, "rb");
    if (!f) return pfail(SCAN_EINVAL, "cannot open checkpoint");
    uint32_t hdr[4] = {0, 0, 0, 0};
    std::vector<float> h(pl->nparams);
    bool ok = std::fread(hdr, sizeof hdr, 1, f) == 1 && hdr[0] == kCkptMagic && hdr[1] == kCkptVersion &&
              hdr[2] == static_cast<uint32_t>(pl->S) && hdr[3] == pl->nparams &&
              std::fread(h.data(), sizeof(float), h.size(), f) == h.size();
    std::fclose(f);
    if (!ok) return pfail(SCAN_EINVAL, "checkpoint header or size does not match this planner");
    return scan_planner_set_params(pl, h.data());
}

}  // extern "C"
