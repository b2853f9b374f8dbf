// Instantiates the scan kernels for widths GB_BLO..GB_BHI (set by the build,
// one object per range so the ranges compile in parallel) and exposes one
// launcher per range.
#include <algorithm>
#include <atomic>

#include "scan_kernels.cuh"

#ifndef GB_BLO
#error "GB_BLO / GB_BHI must be defined by the build"
#endif

namespace gb {
namespace {

// cudaFuncSetAttribute once per (kernel, device): every instantiation may use
// up to the whole shared-memory budget; each launch passes its own size.
template <auto KERNEL>
cudaError_t configure_smem()
{
    static std::atomic<unsigned long long> done_mask{0ull};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done_mask.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(KERNEL), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kSmemMax);
    if (e == cudaSuccess) done_mask.fetch_or(bit, std::memory_order_acq_rel);
    return e;
}

// A full scan with at most one tile per warp of the full grid is cut finer, into
// tiles of one warp step: on one CTA, whose sum needs no global round trip, while 16
// warps hold it (n = 10^4: 2.0-2.7 us a launch against 4.7-5.7 on all SMs), then in
// CTAs of 8 warps until they cover the SMs, then of as many as that takes.  (CTAs of
// one warp: the last CTA's fold of their sums took a round trip per 32 of them.)
inline void fit_small(const ScanParams& p, uint32_t step, LaunchShape& sh, int& grid)
{
    const uint64_t blocks = p.n >> 10;
    const uint64_t sms = static_cast<uint64_t>(grid), most = static_cast<uint64_t>(sh.warps);
    const uint64_t room = sms * most;
    if (blocks > room * static_cast<uint64_t>(sh.tile_blocks)) return;
    const uint64_t tb = std::max<uint64_t>(step, (blocks + room * step - 1) / (room * step) * step);
    const uint64_t need = (blocks + tb - 1) / tb + ((p.n & 1023u) ? 1u : 0u);  // the tail takes a warp of its own
    const uint64_t warps =
        need <= most ? std::max<uint64_t>(need, 1u)
                     : std::min<uint64_t>(std::max<uint64_t>((need + sms - 1) / sms, std::min<uint64_t>(8u, most)), most);
    sh.tile_blocks = static_cast<int>(tb);
    sh.stages = 1;
    sh.warps = static_cast<int>(warps);
    grid = static_cast<int>(std::min<uint64_t>((need + warps - 1) / warps, sms));
    if (grid < 1) grid = 1;
}

template <int B, auto KERNEL, uint32_t SMALL_STEP = 0>
cudaError_t launch_one(const ScanParams& p, LaunchShape sh, int grid, cudaStream_t st, bool overlap = false)
{
    if (const cudaError_t e = configure_smem<KERNEL>(); e != cudaSuccess) return e;
    ScanParams q = p;
    if constexpr (SMALL_STEP != 0) fit_small(p, SMALL_STEP, sh, grid);
    q.tile_blocks = static_cast<uint32_t>(sh.tile_blocks);
    q.stages = static_cast<uint32_t>(sh.stages);
    const uint32_t smem = pipe_smem_bytes(B, sh.warps, sh.stages, sh.tile_blocks);
    // an overlapping launch's CTAs arrive as SMs come free: one per SM
    const uint32_t least = overlap ? 116u * 1024u : 0u;
    return launch_overlapped(KERNEL, grid, sh.warps * 32, smem > least ? smem : least, st, overlap, q);
}

// Full scans.  Bit-sliced widths take one lane per thread and one vote per two
// blocks: every vote form and geometry of their shape runs the same kernel.  The
// others: the 16-warp-bound instantiation for CTAs above 8 warps, the 2-lane
// geometry and the branchy vote form the shape asks for.
template <int B, bool BRANCHY>
cudaError_t launch_full(const ScanParams& p, const LaunchShape& sh, int grid, cudaStream_t st)
{
    if constexpr (sliced(B, BRANCHY)) {
        return launch_one<B, k_scan_full<B, BRANCHY, kLayLanes, 16>, 1>(p, filled(B, sh), grid, st);
    } else {
        constexpr uint32_t kStep = default_lpt(B);
        if constexpr (!BRANCHY && B <= 16) {  // the 2-lane geometry: 16-warp bound only
            if (sh.vec_lanes == 2) return launch_one<B, k_scan_full<B, false, kLayLanes, 16, 0, 2>, 2>(p, sh, grid, st);
        }
        if (sh.vec_lanes != 0 && sh.vec_lanes != default_lpt(B)) return cudaErrorInvalidValue;
        const bool w16 = sh.warps > 8;
        if constexpr (BRANCHY && B <= 21) {
            // the PTX row vote: the 16-warp bound only (any CTA up to 16 warps)
            if (sh.vote_rows == 3) return launch_one<B, k_scan_full<B, true, kLayLanes, 16, 3>, kStep>(p, sh, grid, st);
            if (sh.vote_rows == 2) return launch_one<B, k_scan_full<B, true, kLayLanes, 16, 2>, kStep>(p, sh, grid, st);
            if (sh.vote_rows)
                return w16 ? launch_one<B, k_scan_full<B, true, kLayLanes, 16, 1>, kStep>(p, sh, grid, st)
                           : launch_one<B, k_scan_full<B, true, kLayLanes, 8, 1>, kStep>(p, sh, grid, st);
        }
        if constexpr (BRANCHY && branchy_filled(B)) {
            const LaunchShape f = filled(B, sh);
            if (f.warps > 8) return launch_one<B, k_scan_full<B, true, kLayLanes, 16>, kStep>(p, f, grid, st);
        }
        return w16 ? launch_one<B, k_scan_full<B, BRANCHY, kLayLanes, 16>, kStep>(p, sh, grid, st)
                   : launch_one<B, k_scan_full<B, BRANCHY, kLayLanes, 8>, kStep>(p, sh, grid, st);
    }
}

// Full scans of row-major columns.  Small ones are cut into tiles of one step of their
// decode: a block, or where the lane decode takes the blocks directly (b = 16, branch-free)
// its four.  (Single blocks there took the masked path with three of four lanes idle, us per
// scan of 10^4 / 2 M / 3 M values: 6.3 / 7.2 / 7.2, with four 5.1 / 6.3 / 6.3.)
template <int B, bool BRANCHY>
cudaError_t launch_row(const ScanParams& p, const LaunchShape& sh, int grid, cudaStream_t st)
{
    if constexpr (sliced(B, BRANCHY, row_decode(B)) || BRANCHY)
        return launch_one<B, k_scan_full<B, BRANCHY, kLayRow, 16>, 1>(p, filled(B, sh), grid, st);
    else
        return launch_one<B, k_scan_full<B, BRANCHY, kLayRow>, row_decode(B) == kLayLanes ? default_lpt(B) : 1>(p, sh, grid, st);
}

// Zone-skip scans, which start while the filter before them ends (a column without a
// whole block has no filter): bit-sliced ones fill up their shape's warps as full scans do.
template <int B, bool BRANCHY>
cudaError_t launch_queue(const ScanParams& p, const LaunchShape& sh, int grid, cudaStream_t st)
{
    if constexpr (sliced(B, BRANCHY)) return launch_one<B, k_scan_queue<B, BRANCHY, 16>>(p, filled(B, sh), grid, st, p.n >= 1024u);
    else return launch_one<B, k_scan_queue<B, BRANCHY>>(p, sh, grid, st, p.n >= 1024u);
}

template <int B>
cudaError_t launch_b(int op, const ScanParams& p, const LaunchShape& sh, int grid, cudaStream_t st)
{
    if (sh.warps > 8 && op != kOpFullBF && op != kOpFullBR) return cudaErrorInvalidValue;
    switch (op) {
    case kOpFullBF: return launch_full<B, false>(p, sh, grid, st);
    case kOpFullBR: return launch_full<B, true>(p, sh, grid, st);
    case kOpQueueBF: return launch_queue<B, false>(p, sh, grid, st);
    case kOpQueueBR: return launch_queue<B, true>(p, sh, grid, st);
    case kOpZoneBuild: return launch_one<B, k_zonemap_build<B>>(p, sh, grid, st);
    case kOpRowBF: return launch_row<B, false>(p, sh, grid, st);
    case kOpRowBR: return launch_row<B, true>(p, sh, grid, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int LO, int HI>
cudaError_t dispatch_range(int b, int op, const ScanParams& p, const LaunchShape& sh, int grid, cudaStream_t st)
{
    if constexpr (LO > HI) {
        return cudaErrorInvalidValue;
    } else {
        if (b == LO) return launch_b<LO>(op, p, sh, grid, st);
        return dispatch_range<LO + 1, HI>(b, op, p, sh, grid, st);
    }
}

}  // namespace
}  // namespace gb

#define GB_CAT2(a, b, c) a##b##_##c
#define GB_CAT(a, b, c) GB_CAT2(a, b, c)

cudaError_t GB_CAT(gb_launch_range_, GB_BLO, GB_BHI)(int b, int op, const gb::ScanParams& p,
                                                     const gb::LaunchShape& sh, int grid, cudaStream_t st)
{
    return gb::dispatch_range<GB_BLO, GB_BHI>(b, op, p, sh, grid, st);
}
