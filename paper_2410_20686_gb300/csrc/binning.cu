// Tile binning of the depth-sorted items (sm_103a):
//   k_count_blocks  per block of 512 depth-sorted items: number of (tile, item) pairs; the items'
//                   footprint words in depth order
//   k_scan_blocks   exclusive scan of the block totals (one CTA) + capacity check
//   k_emit          the items' (tile id, item) pairs, one per tile a footprint meets, in depth order at
//                   the exclusive-scan offsets, a warp's items together; counts the tile sort's digits;
//                   items with more than 32 tiles or 6 row bands are queued for k_emit_big; pairs beyond
//                   the capacity are dropped (status bit kStCapacity set by k_scan_blocks)
//   k_emit_big      the queued items, one warp each, or several for those of many tiles
//   k_tile_ranges   [start, end) of every tile's run in the tile-sorted pair list
// An item's rect is (ty0 | bands << 16, number of tiles, spans of bands 0 and 1), rect2 the spans
// of bands 2..5; the columns of further bands are recomputed from its records by band_columns
// (odgs_common.cuh), exactly as the preprocess counted them. With truncated lists (saturation.cu) an
// item writes only the pairs of the tiles that keep its depth bucket, compacted in its tile order; the
// scan uses the kept counts.
#include "odgs_common.cuh"
#include "odgs_internal.h"

namespace odgs {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 2;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* s) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long t = 0ull;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s[w];
    __syncthreads();
    return t;
}

// Tiles t of one row run [row + s, row + s + c) (mod tiles_x) with cut[t] >= b, from bucket b's
// prefix counts G over the tiles.
__device__ __forceinline__ uint32_t kept_in_run(const uint32_t* G, uint32_t row, int s, int c, int tiles_x) {
    const int first = min(c, tiles_x - s);
    uint32_t n = G[row + (uint32_t)(s + first)] - G[row + (uint32_t)s];
    if (c > first) n += G[row + (uint32_t)(c - first)] - G[row];
    return n;
}

// Span (start | count << 16) of stored band b < 6, without a dynamically indexed array.
__device__ __forceinline__ uint32_t stored_span(uint4 rc, const uint4* rect2, uint32_t idx, int b) {
    if (b == 0) return rc.z;
    if (b == 1) return rc.w;
    const uint4 r2 = rect2[idx];
    return b == 2 ? r2.x : (b == 3 ? r2.y : (b == 4 ? r2.z : r2.w));
}

// Pairs per block of 512 depth-sorted items. With truncated lists, the kept pairs of each item
// (its tiles whose cut keeps its depth bucket), stored per position for the emission: per row
// band two prefix-count loads, the bands of items with more than six (whose columns are not
// stored) computed by the warp, one band per lane.
__global__ void __launch_bounds__(kScanThreads) k_count_blocks(BinArgs a) {
    __shared__ unsigned long long s[kScanThreads / 32];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t base = blockIdx.x * kScanTile;
    // the tile ranges of this binning start from 0 (k_tile_ranges writes the non-empty ones)
    if (a.ranges_zero)
        for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < a.n_ranges; t += gridDim.x * blockDim.x)
            a.ranges_zero[t] = make_uint2(0u, 0u);
    // culled items end the depth order
    const uint32_t n_vis = a.partition ? (uint32_t)min((unsigned long long)a.n_items, a.hdr->visible) : a.n_items;
    if (base >= n_vis) {
        if (threadIdx.x == 0) a.block_sums[blockIdx.x] = 0ull;
        return;
    }
    unsigned long long c = 0ull;
    for (int i = threadIdx.x; i < kScanTile; i += kScanThreads) {
        const uint32_t k = base + i;
        uint4 rc = make_uint4(0u, 0u, 0u, 0u);
        uint32_t idx = 0u;
        if (k < n_vis) {
            idx = a.sorted_idx[k];
            // idx >= n_items only after a depth sort that gave up (status already set)
            if (idx < a.n_items) rc = a.rect[idx];
            a.srect[k] = rc;
        }
        if (!a.G) {
            c += rc.y;
            continue;
        }
        const int nb = (int)(rc.x >> 16), ty0 = (int)(rc.x & 0xFFFFu);
        const int bk = k < n_vis ? depth_bucket(a.sorted_keys[k], a.base) : 0;
        const uint32_t* G = a.G + (size_t)bk * (a.total_tiles + 1u);
        // every tile of the frame keeps this bucket (the items in front of the first cut, among
        // them the near, large ones with many bands): the whole footprint
        const bool all = rc.y > 0u && G[a.total_tiles] == a.total_tiles;
        uint32_t kept = all ? rc.y : 0u;
        if (rc.y > 0u && !all && nb <= 6) {
            const ViewDev& V = a.views[idx / (uint32_t)a.n_per_view];
            const uint4 r2 = nb > 2 ? a.rect2[idx] : make_uint4(0u, 0u, 0u, 0u);
            for (int b = 0; b < nb; ++b) {
                const uint32_t sp = b == 0 ? rc.z : (b == 1 ? rc.w : (b == 2 ? r2.x : (b == 3 ? r2.y : (b == 4 ? r2.z : r2.w))));
                const uint32_t row = (uint32_t)V.tile_base + (uint32_t)(ty0 + b) * (uint32_t)V.tiles_x;
                if (sp >> 16) kept += kept_in_run(G, row, (int)(sp & 0xFFFFu), (int)(sp >> 16), V.tiles_x);
            }
        }
        // items of more bands (near, large Gaussians, which cluster at the front of the depth
        // order): queued for k_count_big, which spreads them over all warps
        const bool many = rc.y > 0u && !all && nb > 6;
        const unsigned m = __ballot_sync(full, many);
        if (m) {
            uint32_t slot = 0u;
            if (lane == __ffs(m) - 1) slot = atomicAdd(&a.hdr->n_count_big, (uint32_t)__popc(m));
            slot = __shfl_sync(full, slot, __ffs(m) - 1);
            if (many) a.big[slot + __popc(m & ((1u << lane) - 1u))] = make_uint2(k, 0u);
        }
        if (many) continue;  // k_count_big writes its word and adds its pairs to the block's sum
        if (k < n_vis) a.kcount[k] = kept | ((uint32_t)bk << 26);
        c += kept;
    }
    c = block_sum_u64(c, s);
    if (threadIdx.x == 0) a.block_sums[blockIdx.x] = c;
}

// Kept pairs of the queued items of more than six bands, one warp per item (static round robin),
// added to their block's sum.
__global__ void __launch_bounds__(256) k_count_big(BinArgs a) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t nq = a.hdr->n_count_big;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < nq; i += nwarps) {
        const uint32_t k = a.big[i].x;
        const uint32_t idx = a.sorted_idx[k];
        const uint4 rc = a.rect[idx];
        const int bk = depth_bucket(a.sorted_keys[k], a.base);
        const ViewDev& V = a.views[idx / (uint32_t)a.n_per_view];
        const Footprint fp = make_footprint(a.rec_a[idx], a.rec_b[idx]);
        int jlo, jhi;
        footprint_rows(fp, V.H, jlo, jhi);
        const uint32_t* G = a.G + (size_t)bk * (a.total_tiles + 1u);
        const int nb = (int)(rc.x >> 16), ty0 = (int)(rc.x & 0xFFFFu);
        uint32_t tot = 0u;
        for (int gb = 0; gb < nb; gb += 32) {
            const int b = gb + lane;
            int start = 0, cnt = 0;
            if (b < 6) {
                const uint32_t sp = stored_span(rc, a.rect2, idx, b);
                start = (int)(sp & 0xFFFFu);
                cnt = (int)(sp >> 16);
            } else if (b < nb) {
                const int ty = ty0 + b, th = a.tile_h;
                band_columns(fp, max(jlo, ty * th), min(jhi, ty * th + th - 1), V.W, a.tile_w, V.tiles_x, V.model == 0,
                             start, cnt);
            }
            const uint32_t row = (uint32_t)V.tile_base + (uint32_t)(ty0 + b) * (uint32_t)V.tiles_x;
            tot += cnt > 0 ? kept_in_run(G, row, start, cnt, V.tiles_x) : 0u;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(full, tot, o);
        if (lane == 0) {
            a.kcount[k] = tot | ((uint32_t)bk << 26);
            if (tot) atomicAdd(a.block_sums + k / kScanTile, (unsigned long long)tot);
        }
    }
}

// Exclusive scan of nblocks totals in place by one CTA of 1024 threads; returns their sum to every thread.
__device__ __forceinline__ unsigned long long scan_totals(unsigned long long* __restrict__ block_sums, int nblocks) {
    // eight consecutive totals per thread and step: a frame of 8M items has 15.6K of them, which took
    // 34 us with one per thread and 15 us so
    constexpr int kEach = 8;
    __shared__ unsigned long long s_warp[32];
    __shared__ unsigned long long s_carry;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0ull;
    __syncthreads();
    for (int base = 0; base < nblocks; base += 1024 * kEach) {
        const int i0 = base + (int)threadIdx.x * kEach;
        unsigned long long v[kEach], sum = 0ull;
#pragma unroll
        for (int k = 0; k < kEach; ++k) {
            v[k] = i0 + k < nblocks ? block_sums[i0 + k] : 0ull;
            sum += v[k];
        }
        unsigned long long x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(full, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[w] = x;
        __syncthreads();
        if (w == 0) {  // inclusive scan of the warps' sums
            unsigned long long t = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(full, t, o);
                if (lane >= o) t += y;
            }
            s_warp[lane] = t;
        }
        __syncthreads();
        unsigned long long at = s_carry + (w > 0 ? s_warp[w - 1] : 0ull) + x - sum;
#pragma unroll
        for (int k = 0; k < kEach; ++k) {
            if (i0 + k < nblocks) block_sums[i0 + k] = at;
            at += v[k];
        }
        __syncthreads();
        if (threadIdx.x == 0) s_carry += s_warp[31];
        __syncthreads();
    }
    return s_carry;
}

__global__ void __launch_bounds__(1024) k_scan_blocks(unsigned long long* __restrict__ block_sums, int nblocks,
                                                      Header* hdr, unsigned long long capacity,
                                                      uint32_t* __restrict__ key_hist, bool truncate, bool partition) {
    // the tile sort's digit counts, which the emission adds up, start from 0
    for (int i = threadIdx.x; i < 4 * 256; i += blockDim.x) key_hist[i] = 0u;
    const unsigned long long total = scan_totals(block_sums, nblocks);
    if (threadIdx.x == 0) {
        unsigned long long used = total < capacity ? total : capacity;
        hdr->pairs_emitted = used;
        hdr->n_pairs_sort = (uint32_t)used;
        hdr->n_big = 0u;
        hdr->n_huge = 0u;
        hdr->n_count_big = 0u;
        hdr->kept_pairs = truncate ? 1u : 0u;
        hdr->by_item = partition ? 1u : 0u;
        if (total > capacity) atomicOr(&hdr->status, kStCapacity);
    }
}

// ------------------------------------------------------------------ emission
//
// A warp writes its pairs as one sequence: the tiles of its items' row bands (runs of columns), listed
// in shared memory, are taken 32 at a time, a lane each, so that the writes are coalesced and every
// lane has a tile whatever the items' sizes. Pairs of tiles that do not keep the item's depth bucket
// are compacted away by a ballot; the kept ones follow one another in the items' order. The kernels wait
// on memory: the footprint words come in depth order from the count, which gathers them anyway, and the
// lists are 8 bytes a run, so that eight CTAs (20.6 KB of shared memory, 32 registers) fit on an SM. Measured (k_emit + k_emit_big, us) against a
// thread per small item that gathered its word: 3M Gaussians, 8 views of 4096 x 2048, emitted twice
// 2157 + 1397 -> 1126 + 1160; 500K, 16 views 240 + 26 -> 174 + 18; 1M, six views 105 + 19 -> 82 + 16; 1M, one
// view 35 + 36 -> 26 + 40; 100K, one view 25 + 16 -> 13 + 14. The words' copy adds 2 to 27 us to the count.
constexpr int kStoredBands = 6;   // row bands whose spans the preprocess stored
constexpr uint32_t kSmallTiles = 32;  // items of more tiles or bands take a warp of their own (k_emit_big)
// Items of at least kHugeTiles tiles take kHugeParts warps, each a range of their row bands. With a warp per
// item the SMs idled two thirds of k_emit_big's time for the last ones, pole-stretched Gaussians of thousands of
// tiles: 1M Gaussians, one view 41 -> 16 us; 100K 14 -> 8; 3M, eight views emitted twice 1170 -> 865 (with the
// line at 256 tiles 20, 6 and 930 us, at 1024 19, 10 and 885; in four or sixteen parts 17, 8, 874 and 18, 8, 903).
constexpr uint32_t kHugeTiles = 512;
constexpr uint32_t kHugeParts = 8;
constexpr int kRuns = 32 * kStoredBands;  // runs a warp lists

// A run: x = global id of its tile row's first tile, y = first column | lane of its item << 11 | index of
// its first tile in the warp's sequence << 16 (below 2^16: 32 rows of at most 2048 tiles).
__device__ __forceinline__ uint2 make_run(uint32_t row, uint32_t col, int item, uint32_t first) {
    return make_uint2(row, col | ((uint32_t)item << 11) | (first << 16));
}
// Its item: x = item, y = position of a kept pair less its rank among the warp's kept pairs, z = depth bucket
// the tiles have to keep (as int; -1: all do), w = tiles per row of its view.

// Writes the pairs of the warp's nr listed runs (tot tiles), `kept` pairs of its sequence having been
// written before; returns their number after it. Counts the tile-sort digits. Pairs at or beyond the
// capacity are neither written nor counted.
__device__ __forceinline__ uint32_t emit_runs(const EmitArgs& a, const uint2* run, const uint4* items, int nr, int tot,
                                              uint32_t kept, int lane, uint32_t (*s_hist)[256]) {
    const unsigned full = 0xffffffffu, lt = (1u << lane) - 1u;
    int rs = 0;  // run that holds the window's first tile
    for (int g0 = 0; g0 < tot; g0 += 32) {
        // the runs starting inside the window, as a bit mask: a lane's run is rs plus the starts at or
        // before it
        const int nx = rs + 1 + lane;
        const int p = nx < nr ? (int)(run[nx].y >> 16) : 0x7fffffff;  // p > g0
        const unsigned starts = __reduce_or_sync(full, p < g0 + 32 ? (1u << (p - g0)) : 0u);
        const int r = rs + __popc(starts & ((2u << lane) - 1u));
        rs += __popc(__ballot_sync(full, p <= g0 + 32));
        const int g = g0 + lane;
        bool write = g < tot;
        uint32_t key = 0u;
        uint4 it = make_uint4(0u, 0u, 0u, 0u);
        if (write) {
            const uint2 R = run[r];
            it = items[(R.y >> 11) & 31u];
            uint32_t tx = (R.y & 2047u) + ((uint32_t)g - (R.y >> 16));
            if (tx >= it.w) tx -= it.w;
            key = R.x + tx;
            write = (int)it.z < 0 || (int)__ldg(a.cut + key) >= (int)it.z;
        }
        const unsigned km = __ballot_sync(full, write);
        const uint32_t o = it.y + kept + (uint32_t)__popc(km & lt);
        kept += (uint32_t)__popc(km);
        if (write && o < (uint32_t)a.capacity) {
            a.keys[o] = key;
            a.vals[o] = it.x;
            for (int q = 0; q < a.key_passes; ++q) atomicAdd(&s_hist[q][(key >> (8 * q)) & 0xFFu], 1u);
        }
    }
    return kept;
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// The pairs of one item whose first is at position off, by a whole warp: lanes list the spans of 32 row bands
// at a time (the stored ones, further ones recomputed as the preprocess counted them). part of parts: a range
// of its bands, whose pairs follow the kept pairs of the bands before, as the counts counted them.
__device__ __forceinline__ void emit_item_warp(uint32_t idx, uint4 rc, uint32_t off, int bucket, const EmitArgs& a, int lane,
                                               uint2* run, uint4* items, uint32_t (*s_hist)[256], int part, int parts) {
    const unsigned full = 0xffffffffu;
    const ViewDev& V = a.views[idx / (uint32_t)a.n_per_view];
    const int th = a.tile_h, ty0 = (int)(rc.x & 0xFFFFu), nb = (int)(rc.x >> 16);
    const uint4 r2 = nb > 2 ? a.rect2[idx] : make_uint4(0u, 0u, 0u, 0u);
    Footprint fp{};
    int jlo = 0, jhi = -1;
    if (nb > kStoredBands) {
        fp = make_footprint(a.rec_a[idx], a.rec_b[idx]);
        footprint_rows(fp, V.H, jlo, jhi);
    }
    auto span = [&](int b, int& start, int& cnt) {
        if (b < kStoredBands) {
            const uint32_t sp = b == 0 ? rc.z : (b == 1 ? rc.w : (b == 2 ? r2.x : (b == 3 ? r2.y : (b == 4 ? r2.z : r2.w))));
            start = (int)(sp & 0xFFFFu);
            cnt = (int)(sp >> 16);
        } else {
            const int ty = ty0 + b;
            band_columns(fp, max(jlo, ty * th), min(jhi, ty * th + th - 1), V.W, a.tile_w, V.tiles_x, V.model == 0, start, cnt);
        }
    };
    if (lane == 0) items[0] = make_uint4(idx, off, (uint32_t)bucket, (uint32_t)V.tiles_x);
    const int first = nb * part / parts, end = nb * (part + 1) / parts;
    uint32_t kept = 0u;
    for (int b = lane; b < first; b += 32) {
        int start = 0, cnt = 0;
        span(b, start, cnt);
        const uint32_t row = (uint32_t)V.tile_base + (uint32_t)(ty0 + b) * (uint32_t)V.tiles_x;
        if (cnt > 0)
            kept += bucket < 0 ? (uint32_t)cnt
                               : kept_in_run(a.G + (size_t)bucket * (a.total_tiles + 1u), row, start, cnt, V.tiles_x);
    }
    if (first > 0) kept = __reduce_add_sync(full, kept);
    for (int gb = first; gb < end; gb += 32) {
        const int b = gb + lane;
        int start = 0, cnt = 0;
        if (b < end) span(b, start, cnt);
        const uint32_t incl = warp_incl_scan((uint32_t)cnt, lane);
        const unsigned nz = __ballot_sync(full, cnt > 0);
        if (cnt > 0)
            run[__popc(nz & ((1u << lane) - 1u))] = make_run((uint32_t)V.tile_base + (uint32_t)(ty0 + b) * (uint32_t)V.tiles_x,
                                                             (uint32_t)start, 0, incl - (uint32_t)cnt);
        __syncwarp();
        kept = emit_runs(a, run, items, __popc(nz), (int)__shfl_sync(full, incl, 31), kept, lane, s_hist);
        __syncwarp();  // the next bands overwrite the list
    }
}

__device__ __forceinline__ void flush_digits(uint32_t (*s_hist)[256], uint32_t* key_hist, int passes) {
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x) {
        const uint32_t c = s_hist[i >> 8][i & 255];
        if (c) atomicAdd(key_hist + i, c);
    }
}

// 32 registers: at the 40 that the two queues make of it, 3M Gaussians, eight views take 1145 us instead of 1073.
__global__ void __launch_bounds__(kScanThreads, 8) k_emit(EmitArgs a) {
    __shared__ unsigned long long s_warp[kScanThreads / 32];
    __shared__ unsigned long long s_carry;
    __shared__ uint32_t s_hist[4][256];
    __shared__ uint2 s_run[kScanThreads / 32][kRuns];
    __shared__ uint4 s_item[kScanThreads / 32][32];
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const uint32_t base = blockIdx.x * kScanTile;
    for (int i = tid; i < 4 * 256; i += kScanThreads) s_hist[i >> 8][i & 255] = 0u;
    if (tid == 0) s_carry = a.block_offsets[blockIdx.x];
    // the sorts' scratch: the tile sort's for this binning, the depth sort's (done by now) for the next
#pragma unroll
    for (int r = 0; r < 2; ++r)
        for (size_t i = (size_t)blockIdx.x * kScanThreads + tid; i < a.clear_quads[r]; i += (size_t)gridDim.x * kScanThreads)
            a.clear[r][i] = make_uint4(0u, 0u, 0u, 0u);
    // (culled items end both depth orders, so a rebuild need not know which it was)
    const uint32_t n_vis = a.visible_first ? (uint32_t)min((unsigned long long)a.n_items, a.hdr->visible) : a.n_items;
    if (base >= n_vis) return;
    const uint32_t* kcount = a.rebuild && !a.hdr->kept_pairs ? nullptr : a.kcount;
    __syncthreads();
    for (int round = 0; round < kScanItems; ++round) {
        const uint32_t k = base + (uint32_t)(round * kScanThreads + tid);
        const uint32_t idx = k < n_vis ? a.sorted_idx[k] : 0u;
        // as k_count_blocks read it (no tiles for an index past the end, after a depth sort that gave up)
        const uint4 rc = k < n_vis ? a.srect[k] : make_uint4(0u, 0u, 0u, 0u);
        // kept pairs (the scan) and the item's whole footprint (warp or shared emission)
        const uint32_t kw = (kcount && k < n_vis) ? kcount[k] : rc.y;
        const uint32_t cnt = kcount ? (kw & 0x3FFFFFFu) : rc.y;
        const int bk = (kcount && cnt < rc.y) ? (int)(kw >> 26) : -1;
        const int nb = (int)(rc.x >> 16);
        const bool one = cnt > 0u && rc.y <= kSmallTiles && nb <= kStoredBands;
        // block-wide exclusive scan of the counts of this round (items in depth order)
        unsigned long long x = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(full, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[w] = x;
        __syncthreads();
        unsigned long long off = s_carry + x - cnt, tot = 0ull;
        for (int j = 0; j < kScanThreads / 32; ++j) {
            const unsigned long long v = s_warp[j];
            if (j < w) off += v;
            tot += v;
        }
        __syncthreads();
        if (tid == 0) s_carry += tot;
        // positions past the capacity (below 2^30) are never written: clamped to 32 bits
        const uint32_t off32 = (uint32_t)min(off, 1ull << 31);
        // small items: the warp's, as one sequence
        uint4 r2 = make_uint4(0u, 0u, 0u, 0u);
        if (one && nb > 2) r2 = a.rect2[idx];
        const uint32_t sp[kStoredBands] = {rc.z, rc.w, r2.x, r2.y, r2.z, r2.w};
        uint32_t nz = 0u;
        if (one) {
#pragma unroll
            for (int b = 0; b < kStoredBands; ++b) nz += (b < nb && (sp[b] >> 16) != 0u) ? 1u : 0u;
        }
        const uint32_t packed = one ? (nz << 16) | rc.y : 0u;  // runs (at most 192) and tiles (1024)
        const uint32_t incl = warp_incl_scan(packed, lane);
        const uint32_t last = __shfl_sync(full, incl, 31);
        const uint32_t kincl = warp_incl_scan(one ? cnt : 0u, lane);
        if (one) {
            const ViewDev& V = a.views[idx / (uint32_t)a.n_per_view];
            const uint32_t tiles_x = (uint32_t)V.tiles_x;
            const uint32_t row = (uint32_t)V.tile_base + (rc.x & 0xFFFFu) * tiles_x;
            uint32_t r = (incl - packed) >> 16, first = (incl - packed) & 0xFFFFu;
            s_item[w][lane] = make_uint4(idx, off32 - (kincl - cnt), (uint32_t)bk, tiles_x);
#pragma unroll
            for (int b = 0; b < kStoredBands; ++b) {
                if (b < nb && (sp[b] >> 16) != 0u) {
                    s_run[w][r++] = make_run(row + (uint32_t)b * tiles_x, sp[b] & 0xFFFFu, lane, first);
                    first += sp[b] >> 16;
                }
            }
        }
        __syncwarp();
        emit_runs(a, s_run[w], s_item[w], (int)(last >> 16), (int)(last & 0xFFFFu), 0u, lane, s_hist);
        __syncwarp();  // the next round overwrites the lists
        // large items: queued for k_emit_big (whole warps, round robin). Depth order
        // clusters the nearest, largest Gaussians into the first blocks, so serving them here
        // would leave a few warps writing most of the pairs.
        // The queue's end holds, backwards, those of them that take several warps.
        const bool big = cnt > 0u && !one, huge = big && rc.y >= kHugeTiles;
        const unsigned bigm = __ballot_sync(full, big && !huge), hugem = __ballot_sync(full, huge);
        if (bigm | hugem) {  // one reservation per warp and queue
            uint32_t base_slot = 0u;
            if (bigm && lane == __ffs(bigm) - 1) base_slot = atomicAdd(&a.hdr->n_big, (uint32_t)__popc(bigm));
            if (hugem && lane == __ffs(hugem) - 1) base_slot = atomicAdd(&a.hdr->n_huge, (uint32_t)__popc(hugem));
            const uint32_t sb = __shfl_sync(full, base_slot, bigm ? __ffs(bigm) - 1 : 0);
            const uint32_t sh = __shfl_sync(full, base_slot, hugem ? __ffs(hugem) - 1 : 0);
            const unsigned lt = (1u << lane) - 1u;
            if (huge)
                a.big[a.n_items - 1u - sh - __popc(hugem & lt)] = make_uint2(k, off32);
            else if (big)
                a.big[sb + __popc(bigm & lt)] = make_uint2(k, off32);
        }
    }
    flush_digits(s_hist, a.key_hist, a.key_passes);
}

__global__ void __launch_bounds__(256, 4) k_emit_big(EmitArgs a) {
    __shared__ uint32_t s_hist[4][256];
    __shared__ uint2 s_run[8][32];
    __shared__ uint4 s_item[8][1];
    for (int i = threadIdx.x; i < 4 * 256; i += blockDim.x) s_hist[i >> 8][i & 255] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t n_parts = a.hdr->n_huge * kHugeParts, n_all = n_parts + a.hdr->n_big;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const bool kept = a.kcount && !(a.rebuild && !a.hdr->kept_pairs);
    // static round-robin over the parts of the huge items, then the others: no shared counter to contend on
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n_all; i += nwarps) {
        const bool huge = i < n_parts;
        const uint2 e = a.big[huge ? a.n_items - 1u - i / kHugeParts : i - n_parts];
        const uint32_t idx = a.sorted_idx[e.x];
        const uint4 rc = a.srect[e.x];
        int bucket = -1;
        if (kept) {
            const uint32_t kw = a.kcount[e.x];
            if ((kw & 0x3FFFFFFu) < rc.y) bucket = (int)(kw >> 26);
        }
        emit_item_warp(idx, rc, e.y, bucket, a, lane, s_run[w], s_item[w], s_hist, huge ? (int)(i % kHugeParts) : 0,
                       huge ? (int)kHugeParts : 1);
        __syncwarp();
    }
    flush_digits(s_hist, a.key_hist, a.key_passes);
}

// ------------------------------------------------------------------ visible items first
//
// Perspective frames cull most (view, Gaussian) items (a cube map's face sees a sixth of the scene), and
// every pass of the depth sort would carry them. The items are partitioned first, stably: the
// visible ones, which alone are sorted, then the culled ones in item order, as the whole sort would leave
// them. 1M Gaussians on six faces (1.1M of 6M items visible): depth sort 204 -> 63 us with 27 us of partition,
// pair count 81 -> 33, emission 80 -> 27; the step 2080 -> 1837 us.
constexpr int kPartThreads = 256, kPartItems = 8, kPartTile = kPartThreads * kPartItems;

__global__ void __launch_bounds__(kPartThreads) k_visible_count(const uint32_t* __restrict__ keys, uint32_t n,
                                                                unsigned long long* __restrict__ block_sums) {
    __shared__ int s_count[kPartThreads / 32];
    const uint32_t base = blockIdx.x * (uint32_t)kPartTile;
    int c = 0;
#pragma unroll
    for (int i = 0; i < kPartItems; ++i) {
        const uint32_t k = base + (uint32_t)(i * kPartThreads) + threadIdx.x;
        c += __popc(__ballot_sync(0xffffffffu, k < n && keys[k] != 0xFFFFFFFFu));
    }
    if ((threadIdx.x & 31) == 0) s_count[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kPartThreads / 32; ++w) t += s_count[w];
        block_sums[blockIdx.x] = (unsigned long long)t;
    }
}

__global__ void __launch_bounds__(1024) k_visible_scan(unsigned long long* __restrict__ block_sums, int nblocks, uint32_t n,
                                                       Header* hdr, const uint32_t* __restrict__ hist,
                                                       uint32_t* __restrict__ ohist) {
    const uint32_t total = (uint32_t)scan_totals(block_sums, nblocks);
    if (threadIdx.x == 0) hdr->n_visible_sort = total;
    // a culled item's key is all ones: it counted once in the last digit of every pass
    ohist[threadIdx.x] = hist[threadIdx.x] - ((threadIdx.x & 255u) == 255u ? n - total : 0u);
}

__global__ void __launch_bounds__(kPartThreads) k_partition(const uint32_t* __restrict__ keys, uint32_t n,
                                                            const unsigned long long* __restrict__ block_sums,
                                                            const Header* __restrict__ hdr, uint32_t* __restrict__ okeys,
                                                            uint32_t* __restrict__ ovals) {
    __shared__ uint32_t s_count[kPartItems][kPartThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t base = blockIdx.x * (uint32_t)kPartTile;
    uint32_t key[kPartItems];
    unsigned m[kPartItems];
#pragma unroll
    for (int i = 0; i < kPartItems; ++i) {
        const uint32_t k = base + (uint32_t)(i * kPartThreads) + threadIdx.x;
        key[i] = k < n ? keys[k] : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int i = 0; i < kPartItems; ++i) {
        m[i] = __ballot_sync(0xffffffffu, key[i] != 0xFFFFFFFFu);
        if (lane == 0) s_count[i][w] = (uint32_t)__popc(m[i]);
    }
    __syncthreads();
    uint32_t vis = (uint32_t)block_sums[blockIdx.x];  // visible items before the warp's items of round i
    const uint32_t n_vis = hdr->n_visible_sort;
#pragma unroll
    for (int i = 0; i < kPartItems; ++i) {
        uint32_t before = vis;
#pragma unroll
        for (int q = 0; q < kPartThreads / 32; ++q) {
            const uint32_t c = s_count[i][q];
            before += q < w ? c : 0u;
            vis += c;
        }
        const uint32_t k = base + (uint32_t)(i * kPartThreads) + threadIdx.x;
        const uint32_t rank = before + (uint32_t)__popc(m[i] & ((1u << lane) - 1u));
        if (k < n) {
            const uint32_t o = key[i] != 0xFFFFFFFFu ? rank : n_vis + (k - rank);
            okeys[o] = key[i];
            ovals[o] = k;
        }
    }
}

cudaError_t launch_partition(const uint32_t* keys, uint32_t n, unsigned long long* block_sums, Header* hdr,
                             const uint32_t* hist, uint32_t* ohist, uint32_t* okeys, uint32_t* ovals, cudaStream_t st,
                             int* launches) {
    const int blocks = (int)((n + kPartTile - 1) / kPartTile);
    if (blocks == 0) return cudaSuccess;
    k_visible_count<<<blocks, kPartThreads, 0, st>>>(keys, n, block_sums);
    k_visible_scan<<<1, 1024, 0, st>>>(block_sums, blocks, n, hdr, hist, ohist);
    k_partition<<<blocks, kPartThreads, 0, st>>>(keys, n, block_sums, hdr, okeys, ovals);
    *launches += 3;
    return cudaGetLastError();
}

// [start, end) of every tile's run. A thread takes 4 consecutive keys (one 16-byte load when the
// array is 16-byte aligned) plus the keys on either side.
__global__ void __launch_bounds__(256) k_tile_ranges(const uint32_t* __restrict__ keys, const Header* __restrict__ hdr,
                                                     uint2* __restrict__ ranges, uint32_t total_tiles) {
    const uint32_t n = hdr->n_pairs_sort;
    const uint32_t nq = (n + 3u) / 4u;
    const bool vec = (reinterpret_cast<uintptr_t>(keys) & 15u) == 0u;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < nq; t += gridDim.x * blockDim.x) {
        const uint32_t i0 = 4u * t;
        uint32_t k[4];
        if (vec && i0 + 4u <= n) {
            const uint4 q = *reinterpret_cast<const uint4*>(keys + i0);
            k[0] = q.x; k[1] = q.y; k[2] = q.z; k[3] = q.w;
        } else {
#pragma unroll
            for (int r = 0; r < 4; ++r) k[r] = (i0 + (uint32_t)r < n) ? keys[i0 + r] : 0xFFFFFFFFu;
        }
        uint32_t prev = i0 > 0u ? keys[i0 - 1u] : 0xFFFFFFFFu;
        const uint32_t next = (i0 + 4u < n) ? keys[i0 + 4u] : 0xFFFFFFFFu;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint32_t i = i0 + (uint32_t)r;
            if (i >= n) break;
            const uint32_t kk = k[r];
            const uint32_t kn = r < 3 ? k[r + 1] : next;
            if (kk < total_tiles) {  // false only after a failed sort (status already set)
                if (i == 0u || prev != kk) ranges[kk].x = i;
                if (i + 1u == n || kn != kk) ranges[kk].y = i + 1u;
            }
            prev = kk;
        }
    }
}

int scan_blocks_for(uint32_t n_items) { return (int)((n_items + kScanTile - 1) / kScanTile); }

cudaError_t launch_binning(const BinArgs& a, cudaStream_t st, int* launches) {
    cudaError_t e;
    const int nb = scan_blocks_for(a.n_items);
    if (a.emit_only) {
        if ((e = cudaMemsetAsync(&a.hdr->n_big, 0, 2 * sizeof(uint32_t), st)) != cudaSuccess) return e;
    } else if (nb > 0) {
        // the kept-count queue counter is 0: cleared by the preprocess's setup and by every scan
        BinArgs ca = a;
        if (!a.truncate) ca.G = nullptr;  // whole footprints
        k_count_blocks<<<nb, kScanThreads, 0, st>>>(ca);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        *launches += 1;
        if (a.truncate) {
            k_count_big<<<a.num_sms * 8, 256, 0, st>>>(a);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
            *launches += 1;
        }
    }
    if (!a.emit_only) {
        k_scan_blocks<<<1, 1024, 0, st>>>(a.block_sums, nb, a.hdr, a.capacity, a.key_hist, a.truncate, a.partition);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        *launches += 1;
    }
    if (nb == 0 && (e = cudaMemsetAsync(a.key_hist, 0, sizeof(uint32_t) * 4 * 256, st)) != cudaSuccess) return e;
    if (nb > 0) {
        EmitArgs ea{};
        ea.sorted_idx = a.sorted_idx; ea.srect = a.srect; ea.rect2 = a.rect2; ea.rec_a = a.rec_a; ea.rec_b = a.rec_b; ea.views = a.views;
        ea.n_per_view = a.n_per_view; ea.n_items = a.n_items; ea.tile_w = a.tile_w; ea.tile_h = a.tile_h;
        ea.block_offsets = a.block_sums; ea.capacity = a.capacity; ea.keys = a.keys; ea.vals = a.vals;
        ea.big = a.big; ea.hdr = a.hdr;
        ea.key_hist = a.key_hist; ea.key_passes = a.key_passes;
        ea.kcount = a.truncate || a.emit_only ? a.kcount : nullptr;
        ea.rebuild = a.emit_only;
        ea.visible_first = a.partition || a.emit_only;
        for (int r = 0; r < 2; ++r) { ea.clear[r] = a.clear[r]; ea.clear_quads[r] = a.clear_quads[r]; }
        ea.cut = a.cut;
        ea.G = a.G;
        ea.total_tiles = (uint32_t)a.total_tiles;
        // zeroed by the scan, except when the scan does not run
        if (a.emit_only && (e = cudaMemsetAsync(a.key_hist, 0, sizeof(uint32_t) * 4 * 256, st)) != cudaSuccess) return e;
        k_emit<<<nb, kScanThreads, 0, st>>>(ea);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_emit_big<<<a.num_sms * 8, 256, 0, st>>>(ea);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        *launches += 2;
    }
    return cudaSuccess;
}

cudaError_t launch_tile_ranges(const uint32_t* keys, const Header* hdr, uint2* ranges, int total_tiles,
                               size_t max_pairs, int num_sms, cudaStream_t st, int* launches, bool zeroed) {
    cudaError_t e;
    if (!zeroed && (e = cudaMemsetAsync(ranges, 0, sizeof(uint2) * (size_t)total_tiles, st)) != cudaSuccess) return e;
    if (max_pairs == 0) return cudaSuccess;
    int blocks = (int)min((max_pairs / 4 + 255) / 256, (size_t)num_sms * 16);
    k_tile_ranges<<<max(blocks, 1), 256, 0, st>>>(keys, hdr, ranges, (uint32_t)total_tiles);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace odgs
