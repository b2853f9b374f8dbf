// Instantiates the batched scan kernel for one predicate flavour and a range
// of widths (GB_BATCH_BRANCHY = 0 or 1, GB_BLO..GB_BHI, set by the build, one
// object per range so the ranges compile in parallel) and exposes its launcher.
#include <atomic>

#include "batch_kernels.cuh"

#if !defined(GB_BATCH_BRANCHY) || !defined(GB_BLO) || !defined(GB_BHI)
#error "GB_BATCH_BRANCHY, GB_BLO and GB_BHI must be defined by the build"
#endif

#define GB_CAT3(a, b, c, d) a##b##_##c##_##d
#define GB_NAME(a, b, c, d) GB_CAT3(a, b, c, d)
#if GB_BATCH_BRANCHY
#define GB_BATCH_LAUNCH GB_NAME(gb_launch_batch_br_, GB_BLO, GB_BHI, w)
#else
#define GB_BATCH_LAUNCH GB_NAME(gb_launch_batch_bf_, GB_BLO, GB_BHI, w)
#endif

namespace {

constexpr bool kBr = GB_BATCH_BRANCHY != 0;

constexpr int kLo = GB_BLO;
static_assert(GB_BHI - GB_BLO + 1 == gb::kBatchRange, "one kernel per range of four widths");

}  // namespace

// The groups' columns are all of widths GB_BLO..GB_BHI; CTAs of `warps` warps.
cudaError_t GB_BATCH_LAUNCH(const gb::BatchParams& p, int warps, int grid, cudaStream_t st)
{
    if (warps < 1 || warps > 16 || p.ngroups < 1 || p.ngroups > static_cast<uint32_t>(gb::kBatchRange))
        return cudaErrorInvalidValue;
    for (uint32_t i = 0; i < p.ngroups; ++i)
        if (p.g[i].b < static_cast<uint32_t>(GB_BLO) || p.g[i].b > static_cast<uint32_t>(GB_BHI)) return cudaErrorInvalidValue;
    static std::atomic<unsigned long long> configured{0ull};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    const void* fn = reinterpret_cast<const void*>(gb::k_scan_batch<kBr, kLo>);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, gb::kSmemMax);
        if (e != cudaSuccess) return e;
        // all of the SM's unified memory as shared memory: two CTAs of up to
        // 112 KB of slots each must fit side by side
        e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 static_cast<int>(cudaSharedmemCarveoutMaxShared));
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    const uint32_t smem =
        static_cast<uint32_t>(warps) * (p.warp_bytes + p.stages * gb::kBatchSlotExtra);
    gb::k_scan_batch<kBr, kLo><<<grid, warps * 32, smem, st>>>(p);
    return cudaGetLastError();
}
