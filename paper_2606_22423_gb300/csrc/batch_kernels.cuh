// Batched scan: thousands of columns in one CUDA-graph launch.
//
// The host cuts every column's 1024-value blocks into tiles (per width, the
// most blocks that fill a 6 KB slot in whole warp steps), groups the
// columns by width and numbers each group's tiles consecutively.  A kernel serves
// the groups of up to four neighbouring widths, one width's code at a time: warps
// pop runs of consecutive tile numbers from a group's atomic counter (a host-built
// table gives each run's first tile and column), so a warp usually stays on one
// column for many tiles; each tile is fetched into the warp's slot ring by bulk TMA
// copies and decoded by the single-column scan's code for that width.
// Columns marked for zone skipping test their blocks' (min, max) before the
// copy and fetch only the surviving runs.  A warp keeps running (count, sum)
// totals while the column does not change and adds them to the column's
// result with three atomics when it does.  The frame of reference is applied
// per flush (SUM_v = SUM_u + base*COUNT is linear).
//
// Per tile of four blocks at b = 8 the kernel issues 540 instructions, 470 of them
// decode (690 before whole tiles were one copy and the predicate's keys were made
// once per column: 2^28 values in one column, 68.6 / 57.6 us).
#pragma once
#include "scan_kernels.cuh"

namespace gb {

enum : uint32_t { kColZone = 1u, kColEmpty = 2u };

struct BatchCol {
    const uint32_t* packed;  // lane-interleaved words
    const uint2* zonemap;    // per-block (min, max) of decoded values, or null
    uint64_t n;              // values
    uint32_t b, base;
    uint32_t tile_blocks;    // blocks per tile
    uint32_t tile_begin;     // first tile number of this column in the launch
    uint32_t lo, wm1;        // predicate in code space (width >= 1)
    uint64_t zlo, zhi;       // predicate on decoded values, for zone tests
    uint32_t flags;          // kColZone, kColEmpty
    uint32_t out;            // result slot
};

// One width group of a launch.
struct BatchGroup {
    const BatchCol* cols;
    const uint2* chunks;           // what each pop takes: first tile and its column, and one entry
                                   // past the last; or null: `chunk` tiles per pop, column by search
    unsigned int* head;            // pop counter, zero before the launch
    uint32_t b;                    // width of every column
    uint32_t ncols;
    uint32_t ntiles;
    uint32_t chunk;                // entries of `chunks`, or tiles per pop without them
    uint32_t slot_bytes;           // bytes per slot: the group's tile
    uint32_t cta_end;              // CTAs below this number (and not below the group before's) start here
};

constexpr int kBatchRange = 4;     // widths per kernel, and groups per launch at most

struct BatchParams {
    BatchGroup g[kBatchRange];     // in any order of widths, all within the kernel's range
    uint32_t ngroups;
    unsigned long long* results;   // per output slot: count, sum, blocks, 0
    unsigned int* status;
    uint32_t stages;               // slots per warp (warps per CTA = blockDim.x / 32)
    uint32_t warp_bytes;           // slot bytes per warp: stages of the launch's largest slot
};

// Default batch shape: 8 warps, each with 2 slots of 6 KB, and at most
// kBatchPairSmem of slots per CTA so that two CTAs share an SM (the kernel
// is compiled for 128 registers a thread), usually of different widths.  With one
// CTA per SM the 4096-column workload's replay took 0.97 ms, with two 0.86; 3 or 4
// stages of smaller slots, 4- or 6-warp CTAs and three CTAs per SM were all
// slower.  The shape is a run-time choice per width group; the autotuner may
// replace it.
constexpr int kBatchWarps = 8;
constexpr int kBatchStages = 2;
constexpr int kBatchSlot = 6 * 1024;
constexpr uint32_t kBatchSlotExtra = 8 + 16;   // a slot's barrier and metadata
// Slot bytes of a CTA that leave room for a second one on the SM (228 KB of
// shared memory per SM, 1 KB of it reserved per CTA).
constexpr uint32_t kBatchPairSmem = 112 * 1024;

__host__ __device__ constexpr uint32_t batch_smem_bytes(uint32_t warps, uint32_t stages, uint32_t slot_bytes)
{
    return warps * stages * (slot_bytes + kBatchSlotExtra);
}

// Default blocks per batch tile at width b: as many as fill a 6 KB slot, a
// multiple of the warp step (4 blocks for b <= 16, else 2), at most 64 (the
// keep mask).
__host__ __device__ constexpr uint32_t batch_tile_blocks(uint32_t b)
{
    const uint32_t step = b <= 16 ? 4u : 2u;
    const uint32_t tb = (static_cast<uint32_t>(kBatchSlot) / (128u * b)) / step * step;
    return tb < step ? step : (tb > 64u ? 64u : tb);
}

// Default warps per CTA at width b: 8, fewer where the one-step tiles of the
// widest columns (b = 14..16, 28..32: 7-8 KB) would overflow kBatchPairSmem.
__host__ __device__ constexpr int batch_default_warps(uint32_t b)
{
    const uint32_t per_warp = static_cast<uint32_t>(kBatchStages) * (batch_tile_blocks(b) * 128u * b + kBatchSlotExtra);
    const uint32_t w = kBatchPairSmem / per_warp;
    return w >= static_cast<uint32_t>(kBatchWarps) ? kBatchWarps : static_cast<int>(w);
}
static_assert(batch_default_warps(32) == 6 && batch_default_warps(1) == 8, "default batch CTAs fit two per SM");

struct __align__(8) SlotMeta {
    uint32_t col;     // column index
    uint32_t blocks;  // blocks in the slot, and kSlotTail if the last is the column's partial tail
};
constexpr uint32_t kSlotTail = 0x80000000u;

// All tiles of one group that this warp pops.  One width's code at a time keeps the
// instruction cache warm (warps popping tiles of all 32 widths stalled on
// instruction fetch).  `phase` carries the slots' barrier parities from group to
// group.  Returns false when a bounded wait gave up.
template <bool BRANCHY, int BFIX>
__device__ __forceinline__ bool batch_group(const BatchGroup& P, unsigned long long* results, unsigned int* status,
                                            int kStages, unsigned char* slots, uint64_t* bars, SlotMeta* meta,
                                            uint32_t& phase, int lane)
{
    const uint32_t kSlot = P.slot_bytes;
    // producer cursor (warp-uniform) and the descriptor of its column, kept in
    // registers: a warp's tiles come in runs of one column, so the descriptor
    // and the next column's first tile are loaded once per run, not per tile
    const uint32_t tb = kSlot / (128u * BFIX);  // every column's tiles are cut alike
    uint32_t t_next = 0, t_end = 0, col = 0;
    bool exhausted = false;
    uint32_t pc_id = ~0u, next_begin = 0;
    uint32_t pc_begin = 0, pc_plain = 0, pc_flags = 0;  // tiles below pc_plain: full, copied whole
    const unsigned char* pc_packed = nullptr;
    const uint2* pc_zm = nullptr;
    uint64_t pc_n = 0, pc_zlo = 0, pc_zhi = 0;
    // zone skipping: the keep bits of blocks [zw_begin, zw_begin + zw_span) of the
    // column (one load of zone entries, a lane per block), and the next window's
    // entries, loaded a window ahead
    const uint32_t zw_span = tb <= 32u ? 32u / tb * tb : 0u;
    uint32_t zw_begin = 0xffffffffu, zw_mask = 0u, zn_begin = 0xffffffffu;
    uint2 zn = make_uint2(0u, 0u);
    auto load_col = [&](uint32_t c) {
        const BatchCol* d = P.cols + c;
        pc_packed = reinterpret_cast<const unsigned char*>(d->packed);
        pc_zm = d->zonemap;
        pc_n = d->n;
        pc_begin = d->tile_begin;
        pc_flags = d->flags;
        pc_zlo = d->zlo;
        pc_zhi = d->zhi;
        next_begin = c + 1 < P.ncols ? __ldg(&P.cols[c + 1].tile_begin) : 0xffffffffu;
        pc_plain = pc_flags ? 0u : pc_begin + static_cast<uint32_t>(pc_n >> 10) / tb;
        pc_id = c;
        zw_begin = 0xffffffffu;
        zn_begin = 0xffffffffu;
    };
    const auto zone_entry = [&](uint32_t k, uint32_t nblocks) {
        return k < nblocks ? __ldg(&pc_zm[k]) : make_uint2(0u, 0u);
    };
    const auto zone_keeps = [&](uint2 z) {
        return static_cast<uint64_t>(z.y) >= pc_zlo && static_cast<uint64_t>(z.x) < pc_zhi;
    };
    // Keep bits of the nb (at most 64) blocks from k0.
    auto zone_mask = [&](uint32_t k0, uint32_t nb, uint32_t nblocks) -> uint64_t {
        if (nb > 32u || zw_span == 0u) {
            const uint32_t lo = __ballot_sync(kFull, k0 + lane < nblocks && zone_keeps(zone_entry(k0 + lane, nblocks)));
            const uint32_t k1 = k0 + 32u + static_cast<uint32_t>(lane);
            const uint32_t hi = __ballot_sync(kFull, k1 < nblocks && zone_keeps(zone_entry(k1, nblocks)));
            const uint64_t m = static_cast<uint64_t>(hi) << 32 | lo;
            return nb >= 64u ? m : m & ((1ull << nb) - 1ull);
        }
        if (k0 < zw_begin || k0 + nb > zw_begin + zw_span || zw_begin == 0xffffffffu) {
            const uint2 z = zn_begin == k0 ? zn : zone_entry(k0 + lane, nblocks);
            zw_begin = k0;
            zw_mask = __ballot_sync(kFull, k0 + lane < nblocks && zone_keeps(z));
            zn_begin = k0 + zw_span;
            zn = zone_entry(zn_begin + lane, nblocks);
        }
        const uint32_t m = zw_mask >> (k0 - zw_begin);
        return nb >= 32u ? m : m & ((1u << nb) - 1u);
    };

    // Moves the cursor to a tile of the chunk, or to the next chunk; false when the
    // group has no more work.
    auto refill = [&]() -> bool {
        if (t_next >= t_end) {
            if (exhausted) return false;
            unsigned int start = 0;
            if (lane == 0) start = atomicAdd(P.head, P.chunks ? 1u : P.chunk);
            start = __shfl_sync(kFull, start, 0);
            if (start >= (P.chunks ? P.chunk : P.ntiles)) {
                exhausted = true;
                return false;
            }
            if (P.chunks) {  // host-built table: one load per pop
                const uint2 e = __ldg(&P.chunks[start]);
                t_end = __ldg(&P.chunks[start + 1].x);
                t_next = e.x;
                col = e.y;
            } else {         // binary search over tile_begin
                t_next = start;
                t_end = min(start + P.chunk, P.ntiles);
                uint32_t lo = 0, hi = P.ncols - 1;
                while (lo < hi) {
                    const uint32_t mid = (lo + hi + 1) >> 1;
                    if (__ldg(&P.cols[mid].tile_begin) <= start) lo = mid;
                    else hi = mid - 1;
                }
                col = lo;
            }
            if (col != pc_id) load_col(col);
        }
        while (next_begin <= t_next) load_col(++col);  // the last column's next_begin is past every tile
        return true;
    };

    // Fetch the next tile with a block to read into slot s; false when there is
    // none.  Tiles without one (an empty predicate, no block kept by the zone map)
    // are passed over, a whole run at a time.  meta[s]: the column and the blocks in
    // the slot, the top bit set when the last of them is the column's partial tail.
    auto produce = [&](int s) -> bool {
        unsigned char* dst = slots + static_cast<uint32_t>(s) * kSlot;
#pragma unroll 1
        for (;;) {
            if (t_next >= t_end || next_begin <= t_next) {
                if (!refill()) return false;
            }
            const uint32_t t = t_next++;
            if (t < pc_plain) {  // a whole tile, no zone test: one copy
                if (lane == 0) {
                    meta[s] = SlotMeta{col, tb};
                    fence_proxy_async_smem();
                    mbar_arrive_expect_tx(&bars[s], kSlot);
                    bulk_g2s(dst, pc_packed + static_cast<uint64_t>(t - pc_begin) * kSlot, kSlot, &bars[s]);
                }
                __syncwarp();
                return true;
            }
            if (pc_flags & kColEmpty) {
                t_next = min(t_end, next_begin);
                continue;
            }
            constexpr uint32_t bb = 128u * BFIX;
            const uint32_t nblocks = static_cast<uint32_t>((pc_n + 1023u) >> 10);
            const uint32_t k0 = (t - pc_begin) * tb;
            const uint32_t nb = min(nblocks - k0, tb);
            uint64_t keep = nb >= 64u ? ~0ull : (1ull << nb) - 1ull;
            if (pc_flags & kColZone) {
                keep = zone_mask(k0, nb, nblocks);
                if (!keep) {
                    // on to the tile of the window's next kept block, or past the window
                    if (nb <= 32u && zw_span != 0u) {
                        const uint32_t rest = zw_mask >> (k0 - zw_begin);
                        const uint32_t run = rest ? static_cast<uint32_t>(__ffs(static_cast<int>(rest)) - 1)
                                                  : zw_begin + zw_span - k0;
                        t_next = min(min(t_end, next_begin), t + max(run / tb, 1u));
                    }
                    continue;
                }
            }
            const uint32_t nk = static_cast<uint32_t>(__popcll(keep));
            if (lane == 0) {
                const bool tail = (pc_n & 1023u) && k0 + nb == nblocks && ((keep >> (nb - 1u)) & 1ull);
                meta[s] = SlotMeta{col, nk | (tail ? kSlotTail : 0u)};
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(&bars[s], nk * bb);
                uint64_t rem = keep;
                uint32_t placed = 0;
                while (rem) {
                    const uint32_t first = static_cast<uint32_t>(__ffsll(static_cast<long long>(rem)) - 1);
                    const uint64_t from = rem >> first;
                    const uint32_t len = (~from == 0ull) ? (64u - first)
                                                          : static_cast<uint32_t>(__ffsll(static_cast<long long>(~from)) - 1);
                    bulk_g2s(dst + placed * bb, pc_packed + static_cast<uint64_t>(k0 + first) * bb, len * bb, &bars[s]);
                    placed += len;
                    rem &= (len + first >= 64u) ? 0ull : (~0ull << (first + len));
                }
            }
            __syncwarp();
            return true;
        }
    };

    int produced = 0;
    for (int s = 0; s < kStages; ++s) {
        if (!produce(s)) break;
        ++produced;
    }

    uint64_t cnt = 0, sum = 0, blocks = 0;
    int cur = -1;
    // the consumer's column, loaded when it changes; its keys too are made once per
    // column (for a sliced width some 6 * b operations)
    Keys<BFIX, BRANCHY> keys{};
    uint32_t cc_lo = 0, cc_wm1 = 0, cc_tail = 0;
    uint32_t cur_out = 0, cur_base = 0;
    auto flush = [&]() {
        uint64_t c2 = cnt, s2 = sum;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            c2 += __shfl_xor_sync(kFull, c2, o);
            s2 += __shfl_xor_sync(kFull, s2, o);
        }
        if (lane == 0 && cur >= 0) {
            unsigned long long* r = results + 4u * cur_out;
            if (c2) atomicAdd(&r[0], static_cast<unsigned long long>(c2));
            if (c2) atomicAdd(&r[1], static_cast<unsigned long long>(s2 + static_cast<uint64_t>(cur_base) * c2));
            if (blocks) atomicAdd(&r[2], static_cast<unsigned long long>(blocks));
        }
        cnt = 0;
        sum = 0;
        blocks = 0;
    };

    bool failed = false;
    int it = 0, s = 0;  // s = it mod stages, kept without a division per tile
#pragma unroll 1
    for (; it < produced; ++it, s = (s + 1 == kStages) ? 0 : s + 1) {
        const SlotMeta m = meta[s];
        if (static_cast<int>(m.col) != cur) {
            flush();
            cur = static_cast<int>(m.col);
            const BatchCol* d = P.cols + m.col;
            cc_lo = d->lo;
            cc_wm1 = d->wm1;
            cc_tail = static_cast<uint32_t>(d->n & 1023u);
            keys = make_keys<BFIX, BRANCHY>(cc_lo, cc_wm1);
            cur_out = d->out;
            cur_base = d->base;
        }
        const bool ok = mbar_wait(&bars[s], (phase >> s) & 1u, kWaitLimitNs);
        if (!__all_sync(kFull, ok)) {
            failed = true;
            break;
        }
        phase ^= 1u << s;
        const unsigned char* slot = slots + static_cast<uint32_t>(s) * kSlot;
        const uint32_t nk = m.blocks & ~kSlotTail;
        const bool tail = (m.blocks & kSlotTail) != 0u;
        const uint32_t nfull = tail ? nk - 1u : nk;
        scan_tile<BFIX, BRANCHY>(slot, nfull, lane, keys, cc_lo, cc_wm1, cnt, sum);
        if (tail)
            agg_block_masked<BFIX, 1>(block_rows<BFIX, 1>(slot + nfull * (128u * BFIX), lane), cc_lo, cc_wm1, cnt,
                                      sum, true, cc_tail, lane);
        blocks += nk;
        __syncwarp();
        if (produce(s)) ++produced;
    }
    if (failed) {
        if (lane == 0) atomicOr(status, kErrTimeout);
        // let this warp's copies in flight land before shared memory is released
        for (int j = it; j < produced && j < it + kStages; ++j) {
            const int s = j % kStages;
            mbar_wait(&bars[s], (phase >> s) & 1u, kDrainLimitNs);
            phase ^= 1u << s;
        }
    }
    flush();
    return !failed;
}

// A kernel serves a range of four widths.  Every CTA starts on one of the launch's
// width groups (its share of the CTAs follows its law time) and its warps go on to
// the next when that has no tile left, so that a group finished early -- zone maps
// skipped most of it -- leaves no SM idle, and a batch of all 32 widths takes 12
// launches side by side (widths of one range part where their shapes have fewer warps)
// instead of 32 in chains (each of those cost some 12 us of ramp and drain).  Compiled for CTAs of up to 16 warps, which caps it at 128
// registers a thread: two 8-warp CTAs then fit one SM.
template <bool BRANCHY, int LO>
__global__ void __launch_bounds__(512, 1) k_scan_batch(const __grid_constant__ BatchParams P)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t nwarps = blockDim.x >> 5;
    const int stages = static_cast<int>(P.stages);
    unsigned char* slots = smem + static_cast<size_t>(warp) * P.warp_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(nwarps) * P.warp_bytes) + warp * stages;
    SlotMeta* meta =
        reinterpret_cast<SlotMeta*>(smem + static_cast<size_t>(nwarps) * (P.warp_bytes + 8u * P.stages)) + warp * stages;
    if (lane == 0) {
        for (int s = 0; s < stages; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
    }
    __syncwarp();
    uint32_t first = 0;
    while (first + 1 < P.ngroups && blockIdx.x >= P.g[first].cta_end) ++first;
    uint32_t phase = 0;  // bit s: parity of slot s's next completion
    bool ok = true;
#pragma unroll 1
    for (uint32_t i = 0; i < P.ngroups && ok; ++i) {
        const BatchGroup& g = P.g[first + i < P.ngroups ? first + i : first + i - P.ngroups];
        switch (static_cast<int>(g.b) - LO) {
        case 0: ok = batch_group<BRANCHY, LO>(g, P.results, P.status, stages, slots, bars, meta, phase, lane); break;
        case 1: ok = batch_group<BRANCHY, LO + 1>(g, P.results, P.status, stages, slots, bars, meta, phase, lane); break;
        case 2: ok = batch_group<BRANCHY, LO + 2>(g, P.results, P.status, stages, slots, bars, meta, phase, lane); break;
        case 3: ok = batch_group<BRANCHY, LO + 3>(g, P.results, P.status, stages, slots, bars, meta, phase, lane); break;
        default: break;  // the host groups widths by range
        }
    }
}

}  // namespace gb

// One launcher per flavour and range of four widths (separate objects).
#define GB_DECLARE_BATCH(lo, hi)                                                                                \
    cudaError_t gb_launch_batch_bf_##lo##_##hi##_w(const gb::BatchParams& p, int warps, int grid, cudaStream_t st); \
    cudaError_t gb_launch_batch_br_##lo##_##hi##_w(const gb::BatchParams& p, int warps, int grid, cudaStream_t st);
GB_DECLARE_BATCH(1, 4)
GB_DECLARE_BATCH(5, 8)
GB_DECLARE_BATCH(9, 12)
GB_DECLARE_BATCH(13, 16)
GB_DECLARE_BATCH(17, 20)
GB_DECLARE_BATCH(21, 24)
GB_DECLARE_BATCH(25, 28)
GB_DECLARE_BATCH(29, 32)
#undef GB_DECLARE_BATCH

// The batch kernel over p's groups, all of one range of widths and of CTAs of
// `warps` warps.
inline cudaError_t gb_launch_batch(bool branchy, const gb::BatchParams& p, int warps, int grid, cudaStream_t st)
{
#define GB_RANGE(k, lo, hi)                                                                                       \
    case k:                                                                                                      \
        return branchy ? gb_launch_batch_br_##lo##_##hi##_w(p, warps, grid, st)                                     \
                       : gb_launch_batch_bf_##lo##_##hi##_w(p, warps, grid, st);
    switch (static_cast<int>(p.g[0].b - 1) / gb::kBatchRange) {
        GB_RANGE(0, 1, 4)
        GB_RANGE(1, 5, 8)
        GB_RANGE(2, 9, 12)
        GB_RANGE(3, 13, 16)
        GB_RANGE(4, 17, 20)
        GB_RANGE(5, 21, 24)
        GB_RANGE(6, 25, 28)
        GB_RANGE(7, 29, 32)
    default: return cudaErrorInvalidValue;
    }
#undef GB_RANGE
}
