// Host side of the batched scan: a plan lays out the tiles of many columns,
// keeps a device descriptor table, and records one CUDA graph per plan:
//   descriptors H2D -> reset results/counters -> the width groups' kernels
// (results are copied back to the host after the replay only when a caller
// asks for host results).
// Running the plan again with new predicates only rewrites the pinned
// descriptor table and replays the graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/gbscan.h"
#include "batch_kernels.cuh"

#include "internal.h"

namespace {

scan_status bfail(scan_status s, const char* msg)
{
    gb_set_last_error(msg);
    return s;
}

scan_status bcuda(cudaError_t e, const char* what)
{
    static thread_local char buf[256];
    snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    gb_set_last_error(buf);
    return gb_cuda_status(e);
}

#define BT_CUDA(call)                                 \
    do {                                              \
        cudaError_t e_ = (call);                      \
        if (e_ != cudaSuccess) return bcuda(e_, #call); \
    } while (0)

int batch_grid() { return gb_device_sms(); }


// Control words after the results: one pop counter per width group (u32),
// then the status word at u32 index kMaxGroups.
constexpr size_t kMaxGroups = 64;
constexpr size_t kCtlWords = 40;  // u64 words: 64 + 1 u32 fit in 33
// A group's time on the whole GPU by the bandwidth law, with GB300 figures (copy
// bandwidth 6.7 TB/s; 10 Tvalues/s of bit-sliced decode, 4.3 of direct), in
// microseconds; its packed bytes and values count whole columns (zone skipping
// only shortens it).
double law_us(double bytes, int b)
{
    return std::max(bytes / 6.7e6, bytes * 8.0 / b / (gb::sliced(b, false) ? 10e6 : 4.3e6));
}
// The CTAs that start on a group are in proportion to its law time: two per SM for
// `full` microseconds of it, which is the batch's own time over 1.5 -- so that one
// wave and a half of CTAs hold the whole batch and each pays its ramp once -- and at
// most kLongestUs, so that a large batch's later CTAs even out what zone maps and
// the law get wrong.  1024 columns of 2^29 values in all (all widths), us per replay:
// 261 / 248 / 248 / 256 / 274 for 1 / 1.5 / 2 / 4 / 6 waves; 2048 of 2^31: 859 / 782 /
// 769 / 749 / 740; 64 of 2^26: 66 / 69 / 75 / 87 / 91.
constexpr double kWaves = 1.5;
constexpr double kLongestUs = 110.0;
constexpr double kShortestUs = 5.0;
// A pop is a share 1/(kPopPart * warps) of the group's work left, in units of a full
// tile's time, of which starting a column (its descriptor, a short tile) costs
// about kColumnCost: pops shrink towards the end, where the short columns are.
// (Equal pops of a quarter of a warp's share: 11% slower on the same 1024 columns;
// a least pop of 3 tiles instead of one: 4% slower.)
// Not below what the group's counter can hand out: it serves a pop in about kPopUs, and
// with all warps of the GPU on one group single tiles are decoded as fast as that.  Where
// no zone map is asked the least pop keeps the counter busy half the time at most; where
// one is, the tiles left cluster in few pops, and a longer one costs more than the wait.
// us per replay, least pop of one tile / of this rule / equal pops of at least 4: 4 columns
// of 2^24 values at b = 20 46 / 36 / 37, at b = 8 35.5 / 26 / 26.5, 16 of 2^24 at b = 20
// 86 / 80 / 81; one sorted column of 2^24, zone skipping at 0.3, b = 20 21.0 / 19.4 / 21.9
// (25.6 with the counter idle half the time).
constexpr double kPopPart = 2.0;
constexpr double kColumnCost = 1.5;
constexpr double kPopUs = 1.75e-3;
// The most of a caller's tiles_per_pop: a pop is one warp's work.
constexpr uint32_t kMostTilesPerPop = 1024;
// The graph's descriptor copy and its reset of the results run side by side, but one after
// the other before a single launch with a table up to this size: the copy is short then, and
// a kernel behind one node starts sooner.  us per replay one after the other / side by side,
// columns of 5000 values: 1 column at b = 8 14.1 / 16.3, 64 at b = 20 19.7 / 20.3, 256 at
// b = 5..8 30.9 / 31.5, 384 at b = 8 29.1 / 26.3.  Several launches start in another order
// behind one node: 256 columns of 2^30 values of all widths 424 / 389, 192 of 2^28 130 / 126.
constexpr size_t kSideBySideBytes = 24 * 1024;

}  // namespace

struct scan_batch {
    uint32_t ncols = 0;
    std::vector<const scan_column*> cols;
    std::vector<int> kernel_of;        // 0 branch-free, 1 branchy
    std::vector<uint32_t> zone;        // 1 if the column skips by zone map
    std::vector<uint32_t> slot_of;     // index of the column in the descriptor table
    uint32_t ncol_k[2] = {0, 0};
    uint32_t tiles_per_pop = 0;
    struct Group {
        int kernel, b;
        uint32_t first, count, ntiles, chunk;
        int ctas;            // CTAs that start on this group
        uint32_t chunk_off;  // offset of this group's pops in the chunk table
        gb::LaunchShape shape;  // warps, stages and tile blocks of this width group
        double bytes;           // packed bytes of its columns
        bool zone;              // a column of it skips by zone map
    };
    std::vector<Group> groups;
    struct Launch {  // groups of one flavour, range of widths, warps and stages
        int kernel, warps, stages;
        std::vector<size_t> groups;
    };
    std::vector<Launch> launches;
    uint2* d_chunks = nullptr;  // all groups' pops: first tile and column of each, one past the last
    size_t chunk_cap = 0;
    gb::BatchCol* h_table = nullptr;   // pinned
    gb::BatchCol* d_table = nullptr;
    unsigned long long* d_results = nullptr;  // 4 words per column, then 2 pop counters + status
    scan_result* h_results = nullptr;  // pinned copy of the results
    cudaStream_t capture_stream = nullptr;
    cudaGraphExec_t graph = nullptr;
};

namespace {

// Lay out the tiles for the current strategies: branch-free columns first, and
// within each flavour by width; the groups of four neighbouring widths that share a
// shape's warps and stages go into one launch, whose CTAs each start on one of them,
// so that an SM mostly runs one or two widths' decode code at a time (a kernel whose
// warps all moved through 32 fully unrolled variants thrashed the instruction cache).
scan_status layout(scan_batch* bt)
{
    std::vector<uint32_t> order;
    std::vector<uint32_t> width(bt->ncols);
    std::vector<uint64_t> length(bt->ncols);
    for (uint32_t i = 0; i < bt->ncols; ++i) {
        const uint2* zm = nullptr;
        const uint32_t* pk;
        uint64_t n;
        uint32_t b, base;
        gb_column_view(bt->cols[i], &pk, &n, &b, &base, &zm);
        width[i] = b;
        length[i] = n;
    }
    for (int k = 0; k < 2; ++k)
        for (uint32_t b = 1; b <= 32; ++b)
        {
            const size_t first = order.size();
            for (uint32_t i = 0; i < bt->ncols; ++i)
                if (bt->kernel_of[i] == k && width[i] == b) order.push_back(i);
            // longest first: the short columns, whose starts cost a warp more than
            // their few tiles, come last and in small pops
            std::stable_sort(order.begin() + static_cast<std::ptrdiff_t>(first), order.end(),
                             [&](uint32_t x, uint32_t y) { return length[x] > length[y]; });
        }
    const size_t table_bytes = std::max<size_t>(1, bt->ncols) * sizeof(gb::BatchCol);
    std::memset(bt->h_table, 0, table_bytes);
    bt->ncol_k[0] = bt->ncol_k[1] = 0;
    bt->groups.clear();
    uint32_t group_tiles = 0;
    for (uint32_t j = 0; j < order.size(); ++j) {
        const uint32_t i = order[j];
        const int k = bt->kernel_of[i];
        if (bt->groups.empty() || bt->groups.back().kernel != k ||
            bt->groups.back().b != static_cast<int>(width[i])) {
            scan_batch::Group g{k, static_cast<int>(width[i]), j, 0, 0, 1, 1, 0, {}, 0.0, false};
            g.shape = gb_shape_for(g.b, k == 1 ? gb::kOpBatchBR : gb::kOpBatchBF);
            bt->groups.push_back(g);
            group_tiles = 0;
        }
        const uint2* zm = nullptr;
        const uint32_t* pk;
        uint64_t n;
        uint32_t b, base;
        gb_column_view(bt->cols[i], &pk, &n, &b, &base, &zm);
        gb::BatchCol& d = bt->h_table[j];
        d.packed = pk;
        d.zonemap = zm;
        d.n = n;
        d.b = b;
        d.base = base;
        d.tile_blocks = static_cast<uint32_t>(bt->groups.back().shape.tile_blocks);
        d.tile_begin = group_tiles;  // tile numbers restart in every width group
        d.out = i;
        const uint64_t nblocks = (n + 1023u) >> 10;
        const uint64_t t = (nblocks + d.tile_blocks - 1) / d.tile_blocks;
        if (group_tiles + t > 0xffffffffull) return bfail(SCAN_EINVAL, "too many tiles in one batch");
        group_tiles += static_cast<uint32_t>(t);
        bt->groups.back().bytes += static_cast<double>(nblocks) * 128.0 * b;
        bt->groups.back().zone |= bt->zone[i] != 0u;
        bt->groups.back().count += 1;
        bt->groups.back().ntiles = group_tiles;
        bt->slot_of[i] = j;
        bt->ncol_k[k] += 1;
    }
    if (bt->groups.size() > kMaxGroups) return bfail(SCAN_EINVAL, "too many width groups");
    std::vector<uint2> chunks;
    const uint64_t cap = 2ull * static_cast<uint64_t>(batch_grid());
    double total_us = 0.0;
    for (const auto& g : bt->groups) total_us += law_us(g.bytes, g.b);
    const double full_us = std::max(kShortestUs, std::min(kLongestUs, total_us / kWaves));
    bt->launches.clear();
    for (size_t gi = 0; gi < bt->groups.size(); ++gi) {
        auto& g = bt->groups[gi];
        const uint64_t gw = static_cast<uint64_t>(g.shape.warps);
        const uint64_t by_tiles = (static_cast<uint64_t>(g.ntiles) + gw - 1) / gw;
        const uint64_t by_time =
            static_cast<uint64_t>(std::ceil(static_cast<double>(cap) * law_us(g.bytes, g.b) / full_us));
        g.ctas = static_cast<int>(std::max<uint64_t>(1, std::min({by_tiles, by_time, cap})));
        if (g.ntiles) {
            scan_batch::Launch* at = nullptr;
            for (auto& l : bt->launches) {
                const auto& h = bt->groups[l.groups.front()];
                if (l.kernel == g.kernel && l.warps == g.shape.warps && l.stages == g.shape.stages &&
                    (h.b - 1) / gb::kBatchRange == (g.b - 1) / gb::kBatchRange)
                    at = &l;
            }
            if (!at) {
                bt->launches.push_back({g.kernel, g.shape.warps, g.shape.stages, {}});
                at = &bt->launches.back();
            }
            at->groups.push_back(gi);
        }
        const double warps = static_cast<double>(g.ctas) * static_cast<double>(gw);
        const double least = std::ceil((g.zone ? 1.0 : 2.0) * kPopUs * g.ctas / static_cast<double>(cap) * g.ntiles /
                                       law_us(g.bytes, g.b));
        double left = static_cast<double>(g.ntiles) + kColumnCost * g.count;
        g.chunk_off = static_cast<uint32_t>(chunks.size());
        uint32_t col = g.first, t = 0;
        while (t < g.ntiles) {
            while (col + 1 < g.first + g.count && bt->h_table[col + 1].tile_begin <= t) ++col;
            chunks.push_back(make_uint2(t, col - g.first));
            if (bt->tiles_per_pop) {
                t += std::min({g.ntiles - t, bt->tiles_per_pop, kMostTilesPerPop});
                continue;
            }
            const double want = std::max(least, left / (kPopPart * warps));
            double got = 0.0;
            uint32_t c = col;
            while (t < g.ntiles && got < want) {
                if (bt->h_table[c].tile_begin == t) got += kColumnCost;
                const uint32_t end = c + 1 < g.first + g.count ? bt->h_table[c + 1].tile_begin : g.ntiles;
                const uint32_t take =
                    std::max<uint32_t>(1, static_cast<uint32_t>(std::min<double>(end - t, std::ceil(want - got))));
                const uint32_t n = std::min(take, end - t);
                got += n;
                t += n;
                while (c + 1 < g.first + g.count && bt->h_table[c + 1].tile_begin <= t) ++c;
            }
            left -= got;
        }
        g.chunk = static_cast<uint32_t>(chunks.size()) - g.chunk_off;
        chunks.push_back(make_uint2(g.ntiles, 0));
    }
    if (chunks.size() > bt->chunk_cap) {
        if (bt->d_chunks) cudaFree(bt->d_chunks);
        bt->d_chunks = nullptr;
        bt->chunk_cap = 0;
        BT_CUDA(cudaMalloc(reinterpret_cast<void**>(&bt->d_chunks), chunks.size() * sizeof(uint2)));
        bt->chunk_cap = chunks.size();
    }
    if (!chunks.empty())
        BT_CUDA(cudaMemcpy(bt->d_chunks, chunks.data(), chunks.size() * sizeof(uint2), cudaMemcpyHostToDevice));
    if (bt->graph) {
        cudaGraphExecDestroy(bt->graph);
        bt->graph = nullptr;
    }
    return SCAN_OK;
}

// Enqueues the kernel over `groups` (of one launch).
cudaError_t launch_groups(scan_batch* bt, const std::vector<size_t>& groups, unsigned long long* ctl, cudaStream_t st)
{
    gb::BatchParams p{};
    uint32_t ctas = 0, slot = 0;
    for (const size_t gi : groups) {
        const auto& g = bt->groups[gi];
        gb::BatchGroup& d = p.g[p.ngroups++];
        d.cols = bt->d_table + g.first;
        d.chunks = bt->d_chunks + g.chunk_off;
        d.head = reinterpret_cast<unsigned int*>(ctl) + gi;
        d.b = static_cast<uint32_t>(g.b);
        d.ncols = g.count;
        d.ntiles = g.ntiles;
        d.chunk = g.chunk;
        d.slot_bytes = static_cast<uint32_t>(g.shape.tile_blocks) * 128u * d.b;
        ctas += static_cast<uint32_t>(g.ctas);
        d.cta_end = ctas;
        slot = std::max(slot, d.slot_bytes);
    }
    const auto& g0 = bt->groups[groups.front()];
    p.results = bt->d_results;
    p.status = reinterpret_cast<unsigned int*>(ctl) + kMaxGroups;
    p.stages = static_cast<uint32_t>(g0.shape.stages);
    p.warp_bytes = p.stages * slot;
    return gb_launch_batch(g0.kernel == 1, p, g0.shape.warps, static_cast<int>(ctas), st);
}

scan_status set_strategy(scan_batch* bt, uint32_t i, scan_strategy st)
{
    const uint2* zm = nullptr;
    const uint32_t* pk;
    uint64_t n;
    uint32_t b, base;
    gb_column_view(bt->cols[i], &pk, &n, &b, &base, &zm);
    bt->kernel_of[i] = 0;
    bt->zone[i] = 0;
    switch (st) {
    case SCAN_AUTO:
    case SCAN_BRANCHFREE: break;
    case SCAN_BRANCHY: bt->kernel_of[i] = 1; break;
    case SCAN_ZONE_SKIP_BF: bt->zone[i] = 1; break;
    case SCAN_ZONE_SKIP_BR:
        bt->zone[i] = 1;
        bt->kernel_of[i] = 1;
        break;
    default: return bfail(SCAN_EINVAL, "unknown strategy");
    }
    if (bt->zone[i] && !zm) return bfail(SCAN_EINVAL, "a zone-skip column has no zone map (scan_zonemap_build first)");
    return SCAN_OK;
}

// Write the predicate fields of the pinned descriptor table.
void fill_predicates(scan_batch* bt, const scan_pred* preds)
{
    for (uint32_t i = 0; i < bt->ncols; ++i) {
        gb::BatchCol& d = bt->h_table[bt->slot_of[i]];
        const int64_t lo_v = static_cast<int64_t>(d.base);
        const int64_t hi_v = lo_v + (1ll << d.b);
        const int64_t lo = std::max(preds[i].lo, lo_v);
        const int64_t hi = std::min(preds[i].hi, hi_v);
        d.flags = bt->zone[i] ? gb::kColZone : 0u;
        if (lo >= hi || d.n == 0) {
            d.flags |= gb::kColEmpty;
            d.lo = 0;
            d.wm1 = 0;
            d.zlo = d.zhi = 0;
        } else {
            d.lo = static_cast<uint32_t>(lo - lo_v);
            d.wm1 = static_cast<uint32_t>(hi - lo - 1);
            d.zlo = static_cast<uint64_t>(lo);
            d.zhi = static_cast<uint64_t>(hi);
        }
    }
}

// Planner features, one CTA per column:
//   f0 = b / 32, f1 = log2(max(N, 1)) / 31,
//   f2 = (log10(max(sigma_hat, 1e-5)) + 5) / 5, sigma_hat = matches / values over up to
//        32 evenly spaced blocks (exact integer sample of the true predicate),
//   f3 = clustering c = 1 - mean_k (max_k - min_k + 1) / (colmax - colmin + 1) from the
//        zone map (0 without one): about 0 for shuffled data, about 1 for sorted data.
__global__ void __launch_bounds__(256) k_batch_features(const gb::BatchCol* __restrict__ cols, float* feats)
{
    __shared__ unsigned long long red_a[8], red_b[8];
    __shared__ double red_d[8];
    const gb::BatchCol c = cols[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t nblocks = (c.n + 1023u) >> 10;
    const uint32_t S = static_cast<uint32_t>(nblocks < 32 ? nblocks : 32);
    const uint64_t mask = (c.b == 32) ? 0xffffffffull : ((1ull << c.b) - 1ull);
    unsigned long long match = 0, seen = 0;
    for (uint32_t idx = threadIdx.x; idx < S * 1024u; idx += blockDim.x) {
        const uint32_t j = idx >> 10, pos = idx & 1023u;
        const uint64_t k = static_cast<uint64_t>(j) * nblocks / S;
        if ((k << 10) + pos >= c.n) continue;
        ++seen;
        if (c.flags & gb::kColEmpty) continue;
        const uint32_t l = pos & 31u, row = pos >> 5;
        const uint32_t bit = row * c.b, w = bit >> 5, sh = bit & 31u;
        const uint32_t* blk = c.packed + k * 32u * c.b;
        uint64_t win = __ldg(&blk[32u * w + l]);
        if (sh + c.b > 32u) win |= static_cast<uint64_t>(__ldg(&blk[32u * (w + 1u) + l])) << 32;
        const uint32_t u = static_cast<uint32_t>((win >> sh) & mask);
        if (u - c.lo <= c.wm1) ++match;
    }
    for (int o = 16; o; o >>= 1) {
        match += __shfl_xor_sync(0xffffffffu, match, o);
        seen += __shfl_xor_sync(0xffffffffu, seen, o);
    }
    if (lane == 0) {
        red_a[warp] = match;
        red_b[warp] = seen;
    }
    __syncthreads();
    unsigned long long tm = 0, ts = 0;
    for (int w = 0; w < 8; ++w) {
        tm += red_a[w];
        ts += red_b[w];
    }
    __syncthreads();
    // clustering from the zone map: column range, then the mean relative block range
    double mean_rel = 1.0;
    if (c.zonemap && nblocks) {
        unsigned long long mn = ~0ull, mx = 0;
        for (uint64_t k = threadIdx.x; k < nblocks; k += blockDim.x) {
            const uint2 z = __ldg(&c.zonemap[k]);
            mn = min(mn, static_cast<unsigned long long>(z.x));
            mx = max(mx, static_cast<unsigned long long>(z.y));
        }
        for (int o = 16; o; o >>= 1) {
            mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane == 0) {
            red_a[warp] = mn;
            red_b[warp] = mx;
        }
        __syncthreads();
        unsigned long long cmn = ~0ull, cmx = 0;
        for (int w = 0; w < 8; ++w) {
            cmn = min(cmn, red_a[w]);
            cmx = max(cmx, red_b[w]);
        }
        const double span = static_cast<double>(cmx - cmn + 1ull);
        double acc = 0.0;
        for (uint64_t k = threadIdx.x; k < nblocks; k += blockDim.x) {
            const uint2 z = __ldg(&c.zonemap[k]);
            acc += static_cast<double>(static_cast<unsigned long long>(z.y) - z.x + 1ull) / span;
        }
        for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) red_d[warp] = acc;
        __syncthreads();
        double tot = 0.0;
        for (int w = 0; w < 8; ++w) tot += red_d[w];
        mean_rel = tot / static_cast<double>(nblocks);
    }
    if (threadIdx.x == 0) {
        const double sigma = ts ? static_cast<double>(tm) / static_cast<double>(ts) : 0.0;
        float* f = feats + 4ull * c.out;
        f[0] = static_cast<float>(c.b) / 32.f;
        f[1] = static_cast<float>(log2(c.n > 0 ? static_cast<double>(c.n) : 1.0) / 31.0);
        f[2] = static_cast<float>((log10(sigma > 1e-5 ? sigma : 1e-5) + 5.0) / 5.0);
        f[3] = static_cast<float>(c.zonemap ? 1.0 - mean_rel : 0.0);
    }
}

// Law fallback (Eq. 2 per strategy): the predicted time of strategy s is
//   max(bytes_s / beta, values_s / T_dec[s]); a zone skip reads the zone map
//   plus a fraction phi = min(1, sigma_hat + (1 - c) + 2 / blocks) of the blocks.
//   Strategies: 0 branch-free, 1 branchy, 2 zone-skip branch-free, 3 zone-skip branchy.
//   A zone strategy of a column without a zone map gets a negative time (unavailable).
__device__ void law_seconds(const float* f, const gb::BatchCol& c, float beta, const double (&tdec)[4],
                            double (&t)[4])
{
    const double n = static_cast<double>(c.n), nb = static_cast<double>((c.n + 1023u) >> 10);
    const double bytes = nb * 128.0 * c.b;
    const double sigma = pow(10.0, 5.0 * f[2] - 5.0);
    double phi = sigma + (1.0 - f[3]) + (nb > 0 ? 2.0 / nb : 1.0);
    phi = phi > 1.0 ? 1.0 : phi;
    const bool has_zone = c.zonemap != nullptr;
    for (int s = 0; s < 4; ++s) {
        const bool zone = s >= 2;
        const double rd = zone ? phi * bytes + 8.0 * nb : bytes;
        const double vals = zone ? phi * n : n;
        t[s] = (zone && !has_zone) ? -1.0 : fmax(rd / beta, vals / tdec[s]);
    }
}

__global__ void k_law_choose(const float* __restrict__ feats, const gb::BatchCol* __restrict__ cols,
                             uint32_t ncols, float beta, float t0, float t1, float t2, float t3,
                             int32_t* __restrict__ out)
{
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ncols) return;
    const gb::BatchCol c = cols[j];
    const double tdec[4] = {t0, t1, t2, t3};
    double t[4];
    law_seconds(feats + 4ull * c.out, c, beta, tdec, t);
    int best = 0;
    double bt = 1e300;
    for (int s = 0; s < 4; ++s) {
        if (t[s] < 0.0) continue;
        if (t[s] < bt) {
            bt = t[s];
            best = s;
        }
    }
    out[c.out] = best;
}

// The same law times as natural-log milliseconds, ncols x 4 (row = the
// column's position in the batch); an unavailable strategy gets kLawNoLogMs.
constexpr float kLawNoLogMs = 30.0f;
__global__ void k_law_times(const float* __restrict__ feats, const gb::BatchCol* __restrict__ cols,
                            uint32_t ncols, float beta, float t0, float t1, float t2, float t3,
                            float* __restrict__ out)
{
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= ncols) return;
    const gb::BatchCol c = cols[j];
    const double tdec[4] = {t0, t1, t2, t3};
    double t[4];
    law_seconds(feats + 4ull * c.out, c, beta, tdec, t);
    for (int s = 0; s < 4; ++s)
        out[4ull * c.out + s] = t[s] < 0.0 ? kLawNoLogMs : static_cast<float>(log(t[s] * 1e3 + 1e-9));
}

}  // namespace

extern "C" {

scan_status scan_batch_create(scan_column* const* cols, uint32_t ncols, const scan_strategy* strategies,
                              uint32_t tiles_per_pop, void* stream, scan_batch** out)
{
    (void)stream;
    gb_set_last_error("");
    if (!out || (ncols && !cols)) return bfail(SCAN_EINVAL, "null pointer");
    *out = nullptr;
    for (uint32_t i = 0; i < ncols; ++i) {
        if (!cols[i]) return bfail(SCAN_EINVAL, "a column pointer is NULL");
        const uint32_t* pk;
        const uint2* zm;
        uint64_t n;
        uint32_t b, base;
        if (!gb_column_view(cols[i], &pk, &n, &b, &base, &zm))
            return bfail(SCAN_EINVAL, "batched scans take lane-interleaved columns");
    }
    auto* bt = new (std::nothrow) scan_batch();
    if (!bt) return bfail(SCAN_ENOMEM, "host allocation failed");
    bt->ncols = ncols;
    bt->tiles_per_pop = tiles_per_pop;
    bt->cols.assign(cols, cols + ncols);
    bt->kernel_of.assign(ncols, 0);
    bt->zone.assign(ncols, 0);
    bt->slot_of.assign(ncols, 0);
    for (uint32_t i = 0; i < ncols; ++i) {
        const scan_status s = set_strategy(bt, i, strategies ? strategies[i] : SCAN_BRANCHFREE);
        if (s != SCAN_OK) {
            delete bt;
            return s;
        }
    }
    const size_t table_bytes = std::max<size_t>(1, ncols) * sizeof(gb::BatchCol);
    const size_t res_bytes = (4ull * std::max<uint32_t>(1, ncols) + kCtlWords) * sizeof(unsigned long long);
    cudaError_t e = cudaMallocHost(reinterpret_cast<void**>(&bt->h_table), table_bytes);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&bt->d_table), table_bytes);
    if (e == cudaSuccess) e = cudaMalloc(reinterpret_cast<void**>(&bt->d_results), res_bytes);
    if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&bt->h_results), res_bytes);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&bt->capture_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        scan_batch_destroy(bt);
        return bcuda(e, "batch allocation");
    }
    const scan_status s = layout(bt);
    if (s != SCAN_OK) {
        scan_batch_destroy(bt);
        return s;
    }
    *out = bt;
    return SCAN_OK;
}

scan_status scan_batch_destroy(scan_batch* bt)
{
    if (!bt) return SCAN_OK;
    cudaDeviceSynchronize();
    if (bt->graph) cudaGraphExecDestroy(bt->graph);
    if (bt->capture_stream) cudaStreamDestroy(bt->capture_stream);
    if (bt->h_table) cudaFreeHost(bt->h_table);
    if (bt->h_results) cudaFreeHost(bt->h_results);
    if (bt->d_table) cudaFree(bt->d_table);
    if (bt->d_results) cudaFree(bt->d_results);
    if (bt->d_chunks) cudaFree(bt->d_chunks);
    delete bt;
    return SCAN_OK;
}

scan_status scan_batch_set_strategies(scan_batch* bt, const scan_strategy* strategies)
{
    gb_set_last_error("");
    if (!bt || (bt->ncols && !strategies)) return bfail(SCAN_EINVAL, "null pointer");
    cudaDeviceSynchronize();  // a replay in flight may still read the table
    for (uint32_t i = 0; i < bt->ncols; ++i) {
        const scan_status s = set_strategy(bt, i, strategies[i]);
        if (s != SCAN_OK) return s;
    }
    return layout(bt);
}

scan_status scan_batch_features(scan_batch* bt, const scan_pred* preds, void* stream, float* dev_features)
{
    gb_set_last_error("");
    if (!bt || !dev_features || (bt->ncols && !preds)) return bfail(SCAN_EINVAL, "null pointer");
    if (!bt->ncols) return SCAN_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    BT_CUDA(cudaStreamSynchronize(st));
    fill_predicates(bt, preds);
    BT_CUDA(cudaMemcpyAsync(bt->d_table, bt->h_table, bt->ncols * sizeof(gb::BatchCol), cudaMemcpyHostToDevice, st));
    k_batch_features<<<bt->ncols, 256, 0, st>>>(bt->d_table, dev_features);
    BT_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status scan_batch_law_choose(scan_batch* bt, const float* dev_features, float beta_bytes_per_s,
                                  const float* t_dec_values_per_s, void* stream, int32_t* dev_choice)
{
    gb_set_last_error("");
    if (!bt || !dev_features || !dev_choice || !t_dec_values_per_s) return bfail(SCAN_EINVAL, "null pointer");
    if (!bt->ncols) return SCAN_OK;
    if (!(beta_bytes_per_s > 0.f)) return bfail(SCAN_EINVAL, "beta must be positive");
    for (int s = 0; s < 4; ++s)
        if (!(t_dec_values_per_s[s] > 0.f)) return bfail(SCAN_EINVAL, "every T_dec must be positive");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_law_choose<<<(bt->ncols + 255) / 256, 256, 0, st>>>(dev_features, bt->d_table, bt->ncols, beta_bytes_per_s,
                                                          t_dec_values_per_s[0], t_dec_values_per_s[1],
                                                          t_dec_values_per_s[2], t_dec_values_per_s[3], dev_choice);
    BT_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status scan_batch_law_times(scan_batch* bt, const float* dev_features, float beta_bytes_per_s,
                                 const float* t_dec_values_per_s, void* stream, float* dev_log_ms)
{
    gb_set_last_error("");
    if (!bt || !dev_features || !dev_log_ms || !t_dec_values_per_s) return bfail(SCAN_EINVAL, "null pointer");
    if (!bt->ncols) return SCAN_OK;
    if (!(beta_bytes_per_s > 0.f)) return bfail(SCAN_EINVAL, "beta must be positive");
    for (int s = 0; s < 4; ++s)
        if (!(t_dec_values_per_s[s] > 0.f)) return bfail(SCAN_EINVAL, "every T_dec must be positive");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_law_times<<<(bt->ncols + 255) / 256, 256, 0, st>>>(dev_features, bt->d_table, bt->ncols, beta_bytes_per_s,
                                                         t_dec_values_per_s[0], t_dec_values_per_s[1],
                                                         t_dec_values_per_s[2], t_dec_values_per_s[3], dev_log_ms);
    BT_CUDA(cudaGetLastError());
    return SCAN_OK;
}

scan_status scan_batch_exec(scan_batch* bt, const scan_pred* preds, void* stream, scan_result* host_out,
                            scan_result* dev_out)
{
    gb_set_last_error("");
    if (!bt || (bt->ncols && !preds)) return bfail(SCAN_EINVAL, "null pointer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // the previous replay may still read the pinned table: wait for it
    BT_CUDA(cudaStreamSynchronize(st));
    fill_predicates(bt, preds);
    const size_t table_bytes = std::max<size_t>(1, bt->ncols) * sizeof(gb::BatchCol);
    const size_t res_words = 4ull * std::max<uint32_t>(1, bt->ncols) + kCtlWords;
    unsigned long long* ctl = bt->d_results + 4ull * std::max<uint32_t>(1, bt->ncols);
    if (!bt->graph) {
        // {copy descriptors, reset results and counters, see kSideBySideBytes} -> the
        // launches, side by side: captured on one stream whose dependencies are set by hand
        cudaStream_t cs = bt->capture_stream;
        BT_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        std::vector<cudaGraphNode_t> roots, ends;
        cudaError_t ce = cudaSuccess;
        const auto note = [&](std::vector<cudaGraphNode_t>& into) {  // the node captured last
            cudaStreamCaptureStatus cst;
            const cudaGraphNode_t* deps = nullptr;
            size_t nd = 0;
            if (ce == cudaSuccess) ce = cudaStreamGetCaptureInfo(cs, &cst, nullptr, nullptr, &deps, nullptr, &nd);
            if (ce == cudaSuccess) into.insert(into.end(), deps, deps + nd);
        };
        const auto after = [&](std::vector<cudaGraphNode_t>& nodes) {  // what the next node waits for
            if (ce == cudaSuccess)
                ce = cudaStreamUpdateCaptureDependencies(cs, nodes.data(), nullptr, nodes.size(),
                                                         cudaStreamSetCaptureDependencies);
        };
        ce = cudaMemcpyAsync(bt->d_table, bt->h_table, table_bytes, cudaMemcpyHostToDevice, cs);
        if (bt->launches.size() != 1 || table_bytes > kSideBySideBytes) {
            note(roots);
            std::vector<cudaGraphNode_t> none;
            after(none);
        }
        if (ce == cudaSuccess) ce = cudaMemsetAsync(bt->d_results, 0, res_words * sizeof(unsigned long long), cs);
        note(roots);
        for (const auto& l : bt->launches) {
            after(roots);
            if (ce == cudaSuccess) ce = launch_groups(bt, l.groups, ctl, cs);
            note(ends);
        }
        if (!ends.empty()) after(ends);
        else after(roots);
        cudaGraph_t g = nullptr;
        cudaError_t ec = cudaStreamEndCapture(cs, &g);
        if (ec == cudaSuccess && ce != cudaSuccess) {
            ec = ce;
            if (g) cudaGraphDestroy(g);
            g = nullptr;
        }
        if (ec != cudaSuccess || !g) return bcuda(ec != cudaSuccess ? ec : cudaErrorUnknown, "graph capture");
        const cudaError_t ei = cudaGraphInstantiate(&bt->graph, g, 0);
        cudaGraphDestroy(g);
        if (ei != cudaSuccess) return bcuda(ei, "cudaGraphInstantiate");
    }
    BT_CUDA(cudaGraphLaunch(bt->graph, st));
    if (dev_out)
        BT_CUDA(cudaMemcpyAsync(dev_out, bt->d_results, 4ull * bt->ncols * sizeof(unsigned long long),
                                cudaMemcpyDeviceToDevice, st));
    if (host_out) {  // results and control words back to the host only when asked for
        BT_CUDA(cudaMemcpyAsync(bt->h_results, bt->d_results, res_words * sizeof(unsigned long long),
                                cudaMemcpyDeviceToHost, st));
        BT_CUDA(cudaStreamSynchronize(st));
        const unsigned int status = reinterpret_cast<const unsigned int*>(
            reinterpret_cast<const unsigned long long*>(bt->h_results) + 4ull * std::max<uint32_t>(1, bt->ncols))[kMaxGroups];
        if (status) return bfail(SCAN_ETIMEOUT, "a device-side wait timed out in the batch kernel");
        std::memcpy(host_out, bt->h_results, sizeof(scan_result) * bt->ncols);
    }
    return SCAN_OK;
}

scan_status scan_batch_status(scan_batch* bt, void* stream)
{
    gb_set_last_error("");
    if (!bt) return bfail(SCAN_EINVAL, "batch is NULL");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const unsigned long long* ctl = bt->d_results + 4ull * std::max<uint32_t>(1, bt->ncols);
    unsigned long long* h_ctl = reinterpret_cast<unsigned long long*>(bt->h_results) + 4ull * std::max<uint32_t>(1, bt->ncols);
    BT_CUDA(cudaMemcpyAsync(h_ctl, ctl, kCtlWords * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    BT_CUDA(cudaStreamSynchronize(st));
    if (reinterpret_cast<const unsigned int*>(h_ctl)[kMaxGroups])
        return bfail(SCAN_ETIMEOUT, "a device-side wait timed out in the batch kernel");
    return SCAN_OK;
}

scan_status scan_batch_autotune(scan_batch* bt, const scan_pred* preds, uint32_t reps, void* stream,
                                uint32_t* groups_tuned, float* rule_us, float* tuned_us)
{
    gb_set_last_error("");
    if (!bt || (bt->ncols && !preds)) return bfail(SCAN_EINVAL, "null pointer");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    reps = std::max<uint32_t>(1, std::min<uint32_t>(reps, 100));
    BT_CUDA(cudaStreamSynchronize(st));
    unsigned long long* ctl = bt->d_results + 4ull * std::max<uint32_t>(1, bt->ncols);
    const size_t table_bytes = std::max<size_t>(1, bt->ncols) * sizeof(gb::BatchCol);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    BT_CUDA(cudaEventCreate(&e0));
    BT_CUDA(cudaEventCreate(&e1));
    auto op_of = [](const scan_batch::Group& g) { return g.kernel == 1 ? gb::kOpBatchBR : gb::kOpBatchBF; };
    // Mean time of `reps` launches of group gi alone, with the shapes installed now.
    auto time_group = [&](size_t gi, float* us) -> scan_status {
        scan_status s = layout(bt);
        if (s != SCAN_OK) return s;
        fill_predicates(bt, preds);
        BT_CUDA(cudaMemcpyAsync(bt->d_table, bt->h_table, table_bytes, cudaMemcpyHostToDevice, st));
        unsigned int* head = reinterpret_cast<unsigned int*>(ctl) + gi;
        const std::vector<size_t> alone{gi};
        float total = 0.f;
        for (uint32_t r = 0; r <= reps; ++r) {  // the first launch warms up
            BT_CUDA(cudaMemsetAsync(head, 0, sizeof(unsigned int), st));
            BT_CUDA(cudaEventRecord(e0, st));
            BT_CUDA(launch_groups(bt, alone, ctl, st));
            BT_CUDA(cudaEventRecord(e1, st));
            BT_CUDA(cudaEventSynchronize(e1));
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (r) total += ms;
        }
        *us = total * 1000.f / static_cast<float>(reps);
        return SCAN_OK;
    };
    // Median time of the whole graph (descriptor copy, reset, every group, result
    // copy) over 2 * reps + 1 replays, with the shapes installed now.
    auto time_graph = [&](float* us) -> scan_status {
        scan_status s = layout(bt);
        if (s != SCAN_OK) return s;
        if ((s = scan_batch_exec(bt, preds, stream, nullptr, nullptr)) != SCAN_OK) return s;  // records the graph
        std::vector<float> ts;
        for (uint32_t r = 0; r < 2 * reps + 1; ++r) {
            BT_CUDA(cudaEventRecord(e0, st));
            BT_CUDA(cudaGraphLaunch(bt->graph, st));
            BT_CUDA(cudaEventRecord(e1, st));
            BT_CUDA(cudaEventSynchronize(e1));
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            ts.push_back(ms * 1000.f);
        }
        std::nth_element(ts.begin(), ts.begin() + ts.size() / 2, ts.end());
        *us = ts[ts.size() / 2];
        return SCAN_OK;
    };
    const std::vector<scan_batch::Group> groups = bt->groups;
    for (const auto& g : groups) gb_shape_install(g.b, op_of(g), nullptr, 0.f, 0.f);
    scan_status status = SCAN_OK;
    // 1. screen: each group alone, the rule and every candidate; keep the three fastest
    std::vector<std::vector<gb::LaunchShape>> finalists(groups.size());
    for (size_t gi = 0; gi < groups.size() && status == SCAN_OK; ++gi) {
        const auto& g = groups[gi];
        if (!g.ntiles) continue;
        float rule = 0.f;
        if ((status = time_group(gi, &rule)) != SCAN_OK) break;
        std::vector<std::pair<float, gb::LaunchShape>> timed;
        for (const gb::LaunchShape& c : gb_shape_candidates(g.b, op_of(g))) {
            gb_shape_install(g.b, op_of(g), &c, 0.f, 0.f);
            float us = 0.f;
            if ((status = time_group(gi, &us)) != SCAN_OK) break;
            if (us < rule) timed.push_back({us, c});
        }
        gb_shape_install(g.b, op_of(g), nullptr, 0.f, 0.f);
        std::sort(timed.begin(), timed.end(), [](const auto& x, const auto& y) { return x.first < y.first; });
        for (size_t k = 0; k < timed.size() && k < 3; ++k) finalists[gi].push_back(timed[k].second);
    }
    // 2. the whole replay: the largest groups first, try each group's finalists
    //    with the others fixed and keep one only if the replay gets faster by
    //    more than 0.3% (the replay's run-to-run spread)
    float rule_graph = 0.f, best_graph = 0.f;
    uint32_t tuned = 0;
    if (status == SCAN_OK) status = time_graph(&rule_graph);
    best_graph = rule_graph;
    std::vector<size_t> order(groups.size());
    for (size_t gi = 0; gi < order.size(); ++gi) order[gi] = gi;
    std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) { return groups[x].bytes > groups[y].bytes; });
    for (const size_t gi : order) {
        if (status != SCAN_OK) break;
        const auto& g = groups[gi];
        const gb::LaunchShape* keep = nullptr;
        for (const gb::LaunchShape& c : finalists[gi]) {
            gb_shape_install(g.b, op_of(g), &c, 0.f, 0.f);
            float us = 0.f;
            if ((status = time_graph(&us)) != SCAN_OK) break;
            if (us < best_graph * 0.997f) {
                best_graph = us;
                keep = &c;
            }
        }
        gb_shape_install(g.b, op_of(g), keep, keep ? best_graph : 0.f, keep ? rule_graph : 0.f);
        if (keep) ++tuned;
    }
    if (status == SCAN_OK && tuned) {  // the whole result must beat the rule, measured again
        float again = 0.f, rule_again = 0.f;
        status = time_graph(&again);
        std::vector<gb::LaunchShape> chosen(groups.size());
        for (size_t gi = 0; gi < groups.size(); ++gi) chosen[gi] = gb_shape_for(groups[gi].b, op_of(groups[gi]));
        for (const auto& g : groups) gb_shape_install(g.b, op_of(g), nullptr, 0.f, 0.f);
        if (status == SCAN_OK) status = time_graph(&rule_again);
        if (status == SCAN_OK && again < rule_again) {
            for (size_t gi = 0; gi < groups.size(); ++gi)
                if (chosen[gi].warps != gb_shape_for(groups[gi].b, op_of(groups[gi])).warps ||
                    chosen[gi].stages != gb_shape_for(groups[gi].b, op_of(groups[gi])).stages ||
                    chosen[gi].tile_blocks != gb_shape_for(groups[gi].b, op_of(groups[gi])).tile_blocks)
                    gb_shape_install(groups[gi].b, op_of(groups[gi]), &chosen[gi], again, rule_again);
            best_graph = again;
            rule_graph = rule_again;
        } else {
            tuned = 0;
            best_graph = rule_again;
            rule_graph = rule_again;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (status != SCAN_OK) {
        for (const auto& g : groups) gb_shape_install(g.b, op_of(g), nullptr, 0.f, 0.f);
        layout(bt);
        return status;
    }
    const scan_status ls = layout(bt);  // the installed shapes; the graph is recorded again
    if (ls != SCAN_OK) return ls;
    if (groups_tuned) *groups_tuned = tuned;
    if (rule_us) *rule_us = rule_graph;
    if (tuned_us) *tuned_us = best_graph;
    return SCAN_OK;
}

scan_status scan_batch_run(const scan_column* const* cols, const scan_pred* preds, uint32_t ncols,
                           const scan_strategy* strategies, void* stream, scan_result* host_out)
{
    scan_batch* bt = nullptr;
    scan_status s = scan_batch_create(const_cast<scan_column* const*>(cols), ncols, strategies, 0, stream, &bt);
    if (s != SCAN_OK) return s;
    s = scan_batch_exec(bt, preds, stream, host_out, nullptr);
    if (s == SCAN_OK) cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    scan_batch_destroy(bt);
    return s;
}

}  // extern "C"
