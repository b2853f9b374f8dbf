// Device encoder: plain uint32 values to b-bit codes, lane-interleaved (paper §3's
// transposed layout) or as one row-major stream, one template instantiation per
// width.
//
// Bound: HBM, 4 bytes read and b/8 written per value.  A warp takes one 1024-value
// block; its 32 loads of 128 contiguous bytes are issued together, so a lane
// holds its whole stream (value 32r + lane in row r) in registers and packs it with
// compile-time shifts; the b words go out as b stores of 128 contiguous bytes.  For
// the row-major layout the values are transposed through shared memory first
// (thread t packs values 32t .. 32t + 31, which fill b whole words), and the words
// back, so that loads and stores stay contiguous.  The form before it (a thread per
// output word, width at run time: two divisions, a loop over the word's values and
// 64-bit shifts) took 480 us for 2^27 values at b = 13; this one 106 (7.1 TB/s, its floor), and
// 115 row-major.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "internal.h"
#include "scan_kernels.cuh"

namespace gb {
namespace {

constexpr int kEncWarps = 8;
constexpr int kEncPad = 33;  // words of a transposed row of 32, one of padding

// Word w of the packed stream of codes u[0..31].
template <int B>
__device__ __forceinline__ void pack_codes(const uint32_t (&u)[32], uint32_t (&W)[B])
{
#pragma unroll
    for (int w = 0; w < B; ++w) W[w] = 0u;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const int bit = r * B, w = bit >> 5, s = bit & 31;
        W[w] |= u[r] << s;
        if (s + B > 32) W[w + 1 < B ? w + 1 : w] |= u[r] >> (32 - s);
    }
}

template <int B, bool ROW>
__global__ void __launch_bounds__(kEncWarps * 32) k_encode(const uint32_t* __restrict__ v, uint64_t n, uint32_t base,
                                                           uint32_t* __restrict__ out, unsigned int* status)
{
    constexpr uint32_t kMask = B < 32 ? (1u << (B & 31)) - 1u : 0xffffffffu;
    __shared__ uint32_t stage[ROW ? kEncWarps : 1][ROW ? 32 * kEncPad : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t nblocks = (n + 1023u) >> 10;
    const uint64_t step = static_cast<uint64_t>(gridDim.x) * kEncWarps;
#pragma unroll 1
    for (uint64_t k = static_cast<uint64_t>(blockIdx.x) * kEncWarps + warp; k < nblocks; k += step) {
        const uint32_t* src = v + (k << 10) + lane;
        uint32_t u[32];
        if ((k + 1) << 10 <= n) {
#pragma unroll
            for (int r = 0; r < 32; ++r) u[r] = __ldcs(src + 32 * r);
#pragma unroll
            for (int r = 0; r < 32; ++r) u[r] -= base;
        } else {  // the ragged tail: zero codes past the end
            const uint32_t rem = static_cast<uint32_t>(n - (k << 10));
#pragma unroll
            for (int r = 0; r < 32; ++r) u[r] = 32u * r + lane < rem ? __ldcs(src + 32 * r) - base : 0u;
        }
        // outside [base, base + 2^b) the wrapped difference has a bit above the code's
        uint32_t any = 0u;
#pragma unroll
        for (int r = 0; r < 32; ++r) any |= u[r];
        if (any & ~kMask) {
            atomicOr(status, kErrRange);
#pragma unroll
            for (int r = 0; r < 32; ++r) u[r] &= kMask;
        }
        uint32_t* dst = out + k * 32u * B;
        uint32_t W[B];
        if constexpr (!ROW) {
            pack_codes<B>(u, W);
#pragma unroll
            for (int w = 0; w < B; ++w) __stcs(dst + 32 * w + lane, W[w]);
        } else {
            uint32_t* s = stage[warp];
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 32; ++r) s[r * kEncPad + lane] = u[r];  // row r: values 32r ..
            __syncwarp();
#pragma unroll
            for (int r = 0; r < 32; ++r) u[r] = s[lane * kEncPad + r];  // this thread's values 32*lane ..
            pack_codes<B>(u, W);
            __syncwarp();
            // an odd width's stride already spreads over the banks; an even one's
            // gets a word of padding after every 32
            constexpr int kRow = (B & 1) ? 32 : kEncPad;
#pragma unroll
            for (int w = 0; w < B; ++w) {
                const int i = lane * B + w;
                s[(i >> 5) * kRow + (i & 31)] = W[w];
            }
            __syncwarp();
#pragma unroll
            for (int w = 0; w < B; ++w) __stcs(dst + 32 * w + lane, s[kRow * w + lane]);
        }
    }
}

template <int LO, int HI>
cudaError_t launch(int b, bool row, const uint32_t* v, uint64_t n, uint32_t base, uint32_t* out, unsigned int* status,
                   int grid, cudaStream_t st)
{
    if constexpr (LO > HI) {
        return cudaErrorInvalidValue;
    } else {
        if (b == LO) {
            // at b = 32 the layouts are the same plain array
            if (row && LO < 32) k_encode<LO, true><<<grid, kEncWarps * 32, 0, st>>>(v, n, base, out, status);
            else k_encode<LO, false><<<grid, kEncWarps * 32, 0, st>>>(v, n, base, out, status);
            return cudaGetLastError();
        }
        return launch<LO + 1, HI>(b, row, v, n, base, out, status, grid, st);
    }
}

// Error words of encoder calls in flight: each call owns one from its launch until
// it has read it, so calls on several threads and streams don't meet.  A free word is
// zero, or marked unknown: a call that failed may have left its error in it, and the next
// one to take it clears it first.  (A word allocated per call cost 150 us: the
// stream-ordered pool gives its memory back at every synchronisation.)
constexpr int kErrWords = 64;
__device__ unsigned int g_err_words[kErrWords];
std::atomic<unsigned long long> g_err_used[64];     // per device, a bit per word
std::atomic<unsigned long long> g_err_unknown[64];  // a word's bit changes only in the hands of its owner

int take_word(std::atomic<unsigned long long>& used)
{
    unsigned long long m = used.load(std::memory_order_relaxed);
    for (;;) {
        if (~m == 0ull) return -1;
        int i = 0;
        while ((m >> i) & 1ull) ++i;
        if (used.compare_exchange_weak(m, m | (1ull << i), std::memory_order_acquire)) return i;
    }
}

// Launch, wait, read the error word; clears it again if it was set.
cudaError_t encode_with(unsigned int* word, int b, bool row, const uint32_t* v, uint64_t n, uint32_t base,
                        uint32_t* out, cudaStream_t st, unsigned int* error)
{
    const uint64_t ctas = (((n + 1023u) >> 10) + kEncWarps - 1) / kEncWarps;
    const uint64_t most = 16ull * static_cast<uint64_t>(gb_device_sms());
    cudaError_t e = launch<1, 32>(b, row, v, n, base, out, word, static_cast<int>(ctas < most ? ctas : most), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(error, word, sizeof *error, cudaMemcpyDeviceToHost, st);
    const cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    if (e == cudaSuccess && *error) {
        e = cudaMemsetAsync(word, 0, sizeof *word, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    return e;
}

}  // namespace
}  // namespace gb

cudaError_t gb_encode(int b, bool rowmajor, const uint32_t* values, uint64_t n, uint32_t base, uint32_t* out,
                      cudaStream_t st, unsigned int* error)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::atomic<unsigned long long>& used = gb::g_err_used[dev & 63];
    const int i = gb::take_word(used);
    if (i >= 0) {
        std::atomic<unsigned long long>& unknown = gb::g_err_unknown[dev & 63];
        const unsigned long long bit = 1ull << i;
        void* words = nullptr;
        e = cudaGetSymbolAddress(&words, gb::g_err_words);
        unsigned int* word = static_cast<unsigned int*>(words) + i;
        if (e == cudaSuccess && (unknown.load() & bit)) e = cudaMemsetAsync(word, 0, sizeof *word, st);
        if (e == cudaSuccess) e = gb::encode_with(word, b, rowmajor, values, n, base, out, st, error);
        if (e == cudaSuccess) unknown.fetch_and(~bit);
        else unknown.fetch_or(bit);
        used.fetch_and(~bit, std::memory_order_release);
        return e;
    }
    // more calls in flight than words: one of this call's own
    unsigned int* word = nullptr;
    e = cudaMallocAsync(reinterpret_cast<void**>(&word), sizeof *word, st);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(word, 0, sizeof *word, st);
    if (e == cudaSuccess) e = gb::encode_with(word, b, rowmajor, values, n, base, out, st, error);
    cudaFreeAsync(word, st);
    return e;
}
