// Stable LSD radix sort of 32-bit keys with 32-bit values (sm_103a), used twice per frame:
//   1. (view, Gaussian) items by the bits of their FP32 radial depth   ("sorting by depth",
//      Sec. 3.1), ties kept in item order;
//   2. the (tile, Gaussian) pairs, emitted in depth order, by tile id.
// Together they give every tile its Gaussians in (depth, index) order, the same order as one
// stable sort of 64-bit (tile | depth) keys, with far fewer bytes moved.
//
// The kernels that write the keys count the digits of all passes; each pass is one "onesweep" kernel
// (Adinets & Merrill 2022): a CTA ranks a 2048- or 4096-key tile in shared memory, publishes its
// per-digit counts, obtains the exclusive prefix of all earlier tiles by decoupled look-back, and writes its keys
// digit-run by digit-run (coalesced). The CTAs are persistent (as many as fit on the GPU, each
// claiming tiles in order), so a sort sized for a capacity far above its keys launches no idle
// CTAs. Look-back waits are bounded: a CTA that has read the
// look-back words `wait_limit` times without reaching an inclusive prefix sets kStTimeout in the
// status word and finishes with a partial prefix; its out-of-range writes are skipped, and every
// consumer of the sorted arrays bounds the indices it reads.
#include "odgs_common.cuh"
#include "odgs_internal.h"
#include "per_device.h"

namespace odgs {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItemsMax = 16;  // 4096 keys per CTA for sorts of at least kLargeSort keys, else 2048
// Whole steps of 600K, 800K and 1M Gaussians (a depth sort of as many items) with the line here and at 2^19:
// 923 / 924, 1066 / 1069 and 1142 / 1146 us; 270K in two views 843 / 848
constexpr size_t kLargeSort = 1u << 20;
constexpr int kRadix = 256;
constexpr uint32_t kFlagAgg = 1u << 30;
constexpr uint32_t kFlagPrefix = 2u << 30;
constexpr uint32_t kCountMask = (1u << 30) - 1u;

// Block-wide exclusive scan of one value per thread (256 threads).
__device__ __forceinline__ uint32_t block_excl_scan_256(uint32_t v, uint32_t* s_warp, uint32_t& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    uint32_t wpre = 0, tot = 0;
#pragma unroll
    for (int i = 0; i < kSortWarps; ++i) {
        uint32_t s = s_warp[i];
        if (i < w) wpre += s;
        tot += s;
    }
    total = tot;
    __syncthreads();
    return wpre + x - v;
}

// A look-back word holds its flag and its count, so its store orders nothing else.
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// IMPLIED: where *implied is 1 the values read are dropped: each is its key's place. (A kernel of its own for the
// pass that may need it: a choice at run time in every pass cost a frame of 8 views 25.48 -> 25.75 ms.)
template <int kSortItems, bool IMPLIED>
__global__ void __launch_bounds__(kSortThreads, 4) k_onesweep(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                         uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                         const uint32_t* __restrict__ n_ptr, int shift,
                                                         int bits, const uint32_t* __restrict__ hist,
                                                         uint32_t* lookback, uint32_t* tile_ctr, uint32_t* status,
                                                         uint32_t wait_limit, const uint32_t* implied) {
    extern __shared__ uint2 s_dyn[];
    uint32_t (*s_mask)[kRadix] = reinterpret_cast<uint32_t (*)[kRadix]>(s_dyn);  // [warps] lanes
    uint32_t (*s_cnt)[kRadix] = s_mask + kSortWarps;                             // [warps] counts
    uint32_t* s_keys = reinterpret_cast<uint32_t*>(s_dyn + kSortWarps * kRadix);
    uint32_t* s_vals = s_keys + kSortThreads * kSortItems;
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_digit_excl[kRadix];
    __shared__ uint32_t s_base[kRadix];
    __shared__ uint32_t s_scan[kSortWarps];
    __shared__ uint32_t s_gex[kRadix];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n = *n_ptr;
    const bool by_index = IMPLIED && *implied;
    const uint32_t mask = (1u << bits) - 1u;
    const uint32_t lt = (1u << lane) - 1u;
    // global digit offset of this pass (exclusive scan of the global histogram), the same for
    // every tile
    uint32_t tot;
    s_gex[tid] = block_excl_scan_256(hist[tid], s_scan, tot);

    // Persistent: the grid holds at most the CTAs that fit on the GPU at once (the pair buffer's
    // capacity, which sizes the sort, is far above the pairs a frame keeps), and each CTA claims
    // tiles in order until they run out. A tile waits only on tiles claimed before it, by CTAs
    // that are running, so the look-back always progresses. When the grid has a CTA for every
    // tile, the CTAs' first claims take them all, and a CTA stops after its first tile.
    const uint32_t per_cta = (uint32_t)(kSortThreads * kSortItems);
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(tile_ctr, 1u);
        for (int i = tid; i < kSortWarps * kRadix; i += kSortThreads) s_dyn[i] = make_uint2(0u, 0u);
        __syncthreads();
        const uint32_t tile = s_tile;
        const uint32_t base = tile * per_cta;
        if (base >= n) break;  // CTA-uniform: every tile has been claimed

        uint32_t key[kSortItems], val[kSortItems], rank[kSortItems];
        const uint32_t wbase = base + (uint32_t)warp * (32u * kSortItems);
#pragma unroll
        for (int i = 0; i < kSortItems; ++i) {
            const uint32_t idx = wbase + (uint32_t)i * 32u + (uint32_t)lane;
            const bool valid = idx < n;
            key[i] = valid ? kin[idx] : 0u;
            val[i] = valid ? vin[idx] : 0u;
            if (IMPLIED && by_index) val[i] = idx;
        }
        // stable warp-level ranking: items are ordered by (warp, i, lane).
#pragma unroll
        for (int i = 0; i < kSortItems; ++i) {
            const uint32_t idx = wbase + (uint32_t)i * 32u + (uint32_t)lane;
            const bool valid = idx < n;
            const uint32_t d = (key[i] >> shift) & mask;
            // lanes holding the same digit: each sets its bit in the digit's mask of the warp. A
            // ballot per digit bit took three times the instructions: 23.3M pairs by tile and 6M items
            // by depth, all passes of 8 views, 4293 -> 3520 us; 1M items and 2.3M pairs 138 -> 128 us
            if (valid) atomicOr(&s_mask[warp][d], 1u << lane);
            __syncwarp();
            const uint32_t m = valid ? s_mask[warp][d] : 0u, c = valid ? s_cnt[warp][d] : 0u;
            __syncwarp();
            const uint32_t below = m & lt;
            if (valid && below == 0u) {  // the first of them
                s_mask[warp][d] = 0u;
                s_cnt[warp][d] = c + (uint32_t)__popc(m);
            }
            __syncwarp();
            rank[i] = c + (uint32_t)__popc(below);
        }
        __syncthreads();
        // per digit (one thread each): exclusive prefix over warps, CTA count
        uint32_t cnt = 0;
        {
            const int d = tid;
#pragma unroll
            for (int w = 0; w < kSortWarps; ++w) {
                uint32_t c = s_cnt[w][d];
                s_cnt[w][d] = cnt;
                cnt += c;
            }
        }
        // publish this tile's count for digit tid
        uint32_t* my = lookback + (size_t)tile * kRadix + tid;
        if (tile == 0) {
            st_relaxed(my, kFlagPrefix | cnt);
        } else {
            st_relaxed(my, kFlagAgg | cnt);
        }
        const uint32_t dex = block_excl_scan_256(cnt, s_scan, tot);
        s_digit_excl[tid] = dex;
        // decoupled look-back for digit tid
        uint32_t excl = 0;
        if (tile > 0) {
            int j = (int)tile - 1;
            uint32_t reads = 0;
            bool more = true;
            while (more) {
                // Four words at a time, whose loads overlap. A tile starts some 600 tiles behind the last
                // inclusive prefix's, and the walk, one load's latency a word, was the longest stall; with two
                // words the sorts take 2 % more and with eight 5 %. Together with masks and counts in arrays
                // of their own (all 32 banks instead of the even ones) and plain stores of the look-back
                // words: all passes of 8 views 3560 -> 3217 us, 16 views 627 -> 573 us, 1M items and 2.3M
                // pairs 126 -> 101 us, 100K items and 570K pairs 59 -> 48 us
                uint32_t e[4];
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    e[r] = j - r >= 0 ? ld_volatile(lookback + (size_t)(j - r) * kRadix + tid) : kFlagPrefix;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (!more) break;
                    if (reads++ >= wait_limit) {  // every read counts, so a limit of 0 gives up at once
                        atomicOr(status, kStTimeout);
                        more = false;
                        break;
                    }
                    const uint32_t flag = e[r] & ~kCountMask;
                    if (flag == 0u) {
                        __nanosleep(32);
                        break;
                    }
                    excl += e[r] & kCountMask;
                    more = flag != kFlagPrefix;
                    --j;
                }
            }
            st_relaxed(my, kFlagPrefix | (excl + cnt));
        }
        s_base[tid] = s_gex[tid] + excl - dex;
        __syncthreads();
        // scatter into shared memory in sorted order within the tile
#pragma unroll
        for (int i = 0; i < kSortItems; ++i) {
            const uint32_t idx = wbase + (uint32_t)i * 32u + (uint32_t)lane;
            if (idx < n) {
                const uint32_t d = (key[i] >> shift) & mask;
                const uint32_t pos = s_digit_excl[d] + s_cnt[warp][d] + rank[i];
                s_keys[pos] = key[i];
                s_vals[pos] = val[i];
            }
        }
        __syncthreads();
        const uint32_t count = min(per_cta, n - base);
        for (uint32_t p = tid; p < count; p += kSortThreads) {
            const uint32_t k = s_keys[p];
            const uint32_t d = (k >> shift) & mask;
            const uint32_t dst = s_base[d] + p;
            if (dst < n) {  // only false after a look-back that gave up (status already set)
                kout[dst] = k;
                vout[dst] = s_vals[p];
            }
        }
        if ((n + per_cta - 1) / per_cta <= gridDim.x) break;
        // the next tile's first barrier orders these reads of s_keys, s_vals and s_base before its writes. s_tile,
        // s_mask and s_cnt, which it writes before that barrier, are last read before the one above
    }
}

constexpr size_t onesweep_smem(int items) {
    return kSortWarps * kRadix * sizeof(uint2) + 2 * sizeof(uint32_t) * (size_t)kSortThreads * items;
}

using OnesweepKernel = decltype(&k_onesweep<kSortItemsMax, false>);
static OnesweepKernel onesweep(bool large, bool implied) {
    if (large) return implied ? k_onesweep<kSortItemsMax, true> : k_onesweep<kSortItemsMax, false>;
    return implied ? k_onesweep<kSortItemsMax / 2, true> : k_onesweep<kSortItemsMax / 2, false>;
}

// CTAs of the kernels for large or smaller sorts that fit on an SM of the current device, with all of its shared
// memory for them (with the static arrays the larger tile needs more than the 48 KB of a plain launch); 0 if
// they cannot be launched there.
static int resident_ctas(bool large, size_t smem) {
    int per_sm = 0;
    for (bool implied : {false, true}) {
        const OnesweepKernel k = onesweep(large, implied);
        if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kSortThreads, smem) != cudaSuccess)
            return 0;
    }
    return per_sm;
}

int radix_passes(int bits) { return (bits + 7) / 8; }

// Look-back words for the smaller (2048-key) tile, which needs the most.
size_t radix_lookback_words(size_t max_items) {
    const size_t per = kSortThreads * (kSortItemsMax / 2);
    size_t tiles = (max_items + per - 1) / per;
    return (tiles ? tiles : 1) * kRadix;
}

// Sorts (k[0], v[0]) by key bits [0, bits); returns the buffer index (0 or 1) that holds the
// result. hist: the digit counts of all passes, [passes][256], from the kernels that wrote the keys.
// scratch: tile counters [4] + lookback [radix_lookback_words]. implied: a device word or null; where it is 1,
// v[0] is not read and the values are 0, 1, 2, ... device: the current one (asked for in every sort, it cost an eager
// frame 6 us of host time and more).
cudaError_t launch_radix_sort(uint32_t* k[2], uint32_t* v[2], const uint32_t* n_ptr, size_t max_items, int bits,
                              uint32_t* hist, uint32_t* tile_ctrs, uint32_t* lookback, uint32_t* status, int num_sms,
                              int device, cudaStream_t st, int* result_buf, int* launches, uint32_t wait_limit, int lb_regions,
                              bool cleared, const uint32_t* implied) {
    const int passes = radix_passes(bits);
    *result_buf = 0;
    if (passes == 0 || max_items == 0) return cudaSuccess;
    cudaError_t e;
    // tile counters placed kCtrBytes before the look-back regions are cleared with them
    cleared = cleared && lb_regions >= passes;
    const bool ctr_with_lb = lb_regions >= passes &&
                             reinterpret_cast<uint8_t*>(lookback) == reinterpret_cast<uint8_t*>(tile_ctrs) + kCtrBytes;
    if (!ctr_with_lb && !cleared && (e = cudaMemsetAsync(tile_ctrs, 0, sizeof(uint32_t) * 4, st)) != cudaSuccess) return e;
    const bool large = max_items >= kLargeSort;
    const int per_cta = kSortThreads * (large ? kSortItemsMax : kSortItemsMax / 2);
    const size_t smem = onesweep_smem(large ? kSortItemsMax : kSortItemsMax / 2);
    const size_t lb_words = radix_lookback_words(max_items);
    const int tiles = (int)((max_items + per_cta - 1) / per_cta);
    // persistent CTAs: as many as fit at once, at most one per tile
    static PerDevice resident[2];
    const int res = resident[large ? 1 : 0].get(device, [&] { return resident_ctas(large, smem); });
    if (res <= 0) {
        e = cudaGetLastError();
        return e != cudaSuccess ? e : cudaErrorInvalidConfiguration;
    }
    const int grid = max(min(tiles, res * num_sms), 1);
    int cur = 0;
    // with a look-back region per pass, one memset clears them all; else the one region is
    // cleared before every pass
    const bool regions = lb_regions >= passes;
    if (regions && !cleared && (e = cudaMemsetAsync(ctr_with_lb ? static_cast<void*>(tile_ctrs) : static_cast<void*>(lookback), 0,
                                        (ctr_with_lb ? kCtrBytes : 0) + sizeof(uint32_t) * lb_words * passes, st)) !=
                       cudaSuccess)
        return e;
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        const int pbits = min(8, bits - shift);
        uint32_t* lb = regions ? lookback + (size_t)p * lb_words : lookback;
        if (!regions && (e = cudaMemsetAsync(lb, 0, sizeof(uint32_t) * lb_words, st)) != cudaSuccess) return e;
        onesweep(large, implied && p == 0)<<<grid, kSortThreads, smem, st>>>(
            k[cur], v[cur], k[cur ^ 1], v[cur ^ 1], n_ptr, shift, pbits, hist + p * kRadix, lb, tile_ctrs + p, status,
            wait_limit, implied);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        *launches += 1;
        cur ^= 1;
    }
    *result_buf = cur;
    return cudaSuccess;
}

}  // namespace odgs
