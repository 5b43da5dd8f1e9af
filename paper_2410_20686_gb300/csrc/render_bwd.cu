// Backward alpha blending (reverse of Eq. 3) on ERP tiles (sm_103a).
//
// Same persistent (view, tile) schedule and layout as the forward kernel: PPT pixels of one row per
// thread, as many columns apart as lanes hold a row of the warp's rectangle (four, or all of the tile's row).
// Each pixel starts from its final transmittance and the index after its last blended Gaussian,
// and walks its tile list back to front, recovering T_j = T_{j+1} / (1 - alpha_j). Per blended
// Gaussian it forms
//   dL/drgb = alpha T g,   dL/dalpha = T (rgb . g) - (B . g) / (1 - alpha),
// with g = dL/dC and B the colour blended behind the Gaussian (background included), and from
// dL/dalpha the gradients w.r.t. opacity, the slice-form conic (a, beta, gamma) and ERP mean
// (u, v) through Eq. 2 (zero when alpha was clamped at 0.99). The skip / clamp decisions and alpha are recomputed
// with the forward kernel's exact operation sequence, so they match it bit for bit.
//
// A thread first sums over its PPT pixels, with dp = dL/d(power) and t the pixel's offset from the
// slice centre (the exponent's own variable), dp, dp t and dp t^2 and dL/drgb; with dy the same
// for all of a thread's pixels, these and dy times the first two and dy^2 times the first are the
// nine values (sum dp t gives the mean terms free of the cancellation an image-axis form suffers
// for needle-like Gaussians). The warp sums them over its lanes (warp_reduce_rows4 where four lanes hold
// a pixel row, else a transpose reduction of the nine values), the CTA over its warps in shared memory;
// then one thread per entry forms dL/d(u, v, conic, opacity), which are linear in these sums, and adds
// them to the per-(view, Gaussian) accumulator with three 16-byte vector atomics.
//
// A warp walks only the entries whose footprint meets its pixels and that one of its pixels reached in
// the forward pass: it tests 32 at a time, one per lane, and takes the ballot's bits from the last.
// The kernel is bound by instruction issue. Measured with the walk, the row reduction and the
// exponents formed before the pixels' tests, against a row test of every entry by every warp and the
// reduction of nine values: 1M Gaussians, one 2048 x 1024 view 696 -> 517 us; 500K Gaussians, 16 views
// 4369 -> 3265 us; 3M Gaussians, 8 views of 4096 x 2048 11438 -> 8920 us. The walk alone: 585, 3660 and
// 9920 us; with a mask per pixel slot instead of per warp 597, 3632 and 10865 us. Without a flag set by
// every blending slot: 508, 3210 and 8700 us.
#include "odgs_common.cuh"
#include "odgs_internal.h"

namespace odgs {

// Sum v[0..8] over the warp. Returns the lane's share: value index *vi (valid iff *ok).
__device__ __forceinline__ float warp_reduce9(const float v[9], int lane, int* vi, bool* ok) {
    const unsigned full = 0xffffffffu;
    bool up = lane & 16;
    float w[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const float hi = (k + 5 < 9) ? v[k + 5] : 0.f;
        const float keep = up ? hi : v[k];
        const float send = up ? v[k] : hi;
        w[k] = keep + __shfl_xor_sync(full, send, 16);
    }
    up = lane & 8;
    float x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float hi = (k + 3 < 5) ? w[k + 3] : 0.f;
        const float keep = up ? hi : w[k];
        const float send = up ? w[k] : hi;
        x[k] = keep + __shfl_xor_sync(full, send, 8);
    }
    up = lane & 4;
    float y[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float hi = (k + 2 < 3) ? x[k + 2] : 0.f;
        const float keep = up ? hi : x[k];
        const float send = up ? x[k] : hi;
        y[k] = keep + __shfl_xor_sync(full, send, 4);
    }
    up = lane & 2;
    float z = (up ? y[1] : y[0]) + __shfl_xor_sync(full, up ? y[0] : y[1], 2);
    z += __shfl_xor_sync(full, z, 1);
    const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1, b1 = (lane >> 1) & 1;
    const int idx = 5 * b4 + 3 * b3 + 2 * b2 + b1;
    *vi = idx;
    *ok = ((lane & 1) == 0) && (2 * b2 + b1 < 3 - b3) && (idx < 9);
    return z;
}

// The warp's nine sums when its lanes hold rows of four (lane = 4 row + column): the six per-lane sums
// are added over the four lanes of a row first, the products with dy (one value per row) formed by
// the lane that owns the sum, then the rows are added: 9 shuffles and 13 selects instead of 12 and 22.
// Returns the lane's share: value index row4_index(lane), if not negative.
__device__ __forceinline__ float warp_reduce_rows4(float S0, float S1, float S2, float V0, float V1, float V2, float dy,
                                                   int lane) {
    const unsigned full = 0xffffffffu;
    bool up = lane & 1;
    const float w0 = (up ? V0 : S0) + __shfl_xor_sync(full, up ? S0 : V0, 1);
    const float w1 = (up ? V1 : S1) + __shfl_xor_sync(full, up ? S1 : V1, 1);
    const float w2 = (up ? V2 : S2) + __shfl_xor_sync(full, up ? S2 : V2, 1);
    up = lane & 2;
    const float x0 = (up ? w1 : w0) + __shfl_xor_sync(full, up ? w0 : w1, 2);  // S0, V0, S1, V1
    const float b = w2 + __shfl_xor_sync(full, w2, 2);                         // S2, V2, S2, V2
    const float x1 = dy * x0;
    const float x2 = (lane & 3) == 0 ? dy * x1 : b;
    up = lane & 16;
    const float y0 = (up ? x1 : x0) + __shfl_xor_sync(full, up ? x0 : x1, 16);
    const float y1 = x2 + __shfl_xor_sync(full, x2, 16);
    up = lane & 8;
    float z = (up ? y1 : y0) + __shfl_xor_sync(full, up ? y0 : y1, 8);
    z += __shfl_xor_sync(full, z, 4);
    return z;
}
__device__ __forceinline__ int row4_index(int lane) {
    const int q = lane & 3;
    if (lane & 4) return -1;
    if ((lane & 24) == 0) return q == 0 ? 0 : (q == 1 ? 6 : (q == 2 ? 1 : 7));  // S0, V0, S1, V1
    if ((lane & 24) == 16) return q == 0 ? 4 : (q == 2 ? 3 : -1);               // dy S0, dy S1
    if ((lane & 24) == 8) return q == 0 ? 5 : (q == 1 ? 8 : (q == 2 ? 2 : -1));  // dy^2 S0, V2, S2
    return -1;
}

// A staged entry, 80 bytes apart (conflict-free 16-byte accesses of consecutive entries).
struct StagedBwd {
    float4 pos, con, col;  // Staged's
    float4 ext;            // stage_extent's
    float4 raw;            // a, gamma (slice-form conic), 1 / opacity, item (bits)
};

template <int PPT, bool ROWS4>
__global__ void __launch_bounds__(256) k_render_bwd(BwdArgs a) {
    extern __shared__ float4 smem[];
    const int B = a.batch;
    const int nwarps = blockDim.x >> 5;
    StagedBwd* s_e = reinterpret_cast<StagedBwd*>(smem);
    float* s_fc2 = reinterpret_cast<float*>(s_e + B);
    float* s_red = s_fc2 + B;                                                      // [B][nwarps][9]
    uint32_t* s_got = reinterpret_cast<uint32_t*>(s_red + (size_t)B * nwarps * 9);  // [nwarps][2]: entries a warp's sums are in s_red for
    __shared__ int s_item;
    __shared__ int s_maxn;

    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int tw = a.tile_w;
    const int rw = region_width(tw, a.tile_h, PPT);
    const int tpr = rw / PPT;  // threads per pixel row of the warp's region
    // a thread's PPT pixels are tpr columns apart (interleaved), so a footprint a few pixels wide
    // falls in one of each lane's pixel slots rather than in several
    const int rx0 = (warp % (tw / rw)) * rw, ry0 = (warp / (tw / rw)) * (32 / tpr);
    const int lx0 = rx0 + lane % tpr, ly = ry0 + lane / tpr;
    const int slot4 = row4_index(lane);
    uint32_t evals = 0u;

    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_item = (int)atomicAdd(&a.hdr->work_bwd, 1u);
            s_maxn = 0;
        }
        __syncthreads();
        const int item = s_item;
        if (item >= a.total_tiles) break;
        int v = 0;
        while (v + 1 < a.n_views && a.views[v + 1].tile_base <= item) ++v;
        const ViewDev& V = a.views[v];
        const int lt = item - V.tile_base;
        const int tx = lt % V.tiles_x, ty = lt / V.tiles_x;
        const int x0 = tx * tw;
        const int xp = x0 + lx0, y = ty * a.tile_h + ly;
        const bool inside = y < V.H;
        const float fj = (float)y;
        float fik[PPT];  // column coordinates of the thread's pixels
#pragma unroll
        for (int k = 0; k < PPT; ++k) fik[k] = (float)(xp + k * tpr);
        const uint2 rg = a.ranges[item];
        // entries past the tile's range (possible only when the lists were rebuilt after a sort
        // that gave up, so that they differ from the forward's) stage as never-blending entries
        const uint32_t rlen = rg.y > rg.x ? rg.y - rg.x : 0u;
        const Region reg = make_region(x0 + rx0, rw, ty * a.tile_h + ry0, 32 / tpr);

        float T[PPT], Bg[PPT], g0[PPT], g1[PPT], g2[PPT];
        int nl[PPT];
        int tmax = 0;
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
            T[k] = 1.f; Bg[k] = 0.f; g0[k] = g1[k] = g2[k] = 0.f; nl[k] = 0;
            if (inside) {
                const int pix = y * V.W + xp + k * tpr;
                const int HW = V.W * V.H;
                T[k] = a.T_final[V.pix_base + pix];
                nl[k] = (int)a.n_last[V.pix_base + pix];
                const float* gi = a.dL_dimages[v];
                g0[k] = gi[pix]; g1[k] = gi[HW + pix]; g2[k] = gi[2 * HW + pix];
                if (a.checked) {  // a non-finite gradient value counts as 0 and is reported
                    const bool f0 = isfinite(g0[k]), f1 = isfinite(g1[k]), f2 = isfinite(g2[k]);
                    if (!(f0 && f1 && f2)) {
                        atomicOr(&a.hdr->status, kStNonfinite);
                        g0[k] = f0 ? g0[k] : 0.f; g1[k] = f1 ? g1[k] : 0.f; g2[k] = f2 ? g2[k] : 0.f;
                    }
                }
                Bg[k] = T[k] * (a.bg[0] * g0[k] + a.bg[1] * g1[k] + a.bg[2] * g2[k]);
                tmax = max(tmax, nl[k]);
                evals += (uint32_t)nl[k];
            }
        }
        if (tmax > 0) atomicMax(&s_maxn, tmax);
        __syncthreads();
        const int maxn = s_maxn;
        const int wmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)tmax);  // warp-uniform bound

        for (int hi = maxn; hi > 0; hi -= B) {
            const int lo = max(0, hi - B);
            const int cnt = hi - lo;
            int split = 0;
            for (int j = tid; j < cnt; j += nthr) {
                const uint32_t idx = (uint32_t)(lo + j) < rlen ? a.pair_vals[rg.x + lo + j] : 0xFFFFFFFFu;
                float4 ra, rb, rc;
                gather_records(a.rec_a, a.rec_b, a.rec_c, idx, a.n_items, ra, rb, rc);
                Staged s = stage_entry(ra, rb, rc, x0, tw, V.W, V.model == 0);
                StagedBwd& e = s_e[j];
                e.pos = s.pos;
                e.con = s.con;
                e.col = s.col;
                e.ext = stage_extent(ra, rb, s.col.w <= 1e30f);
                e.raw = make_float4(rb.x, rb.z, ra.w > 0.f ? 1.f / ra.w : 0.f,
                                    __uint_as_float(idx < a.n_items ? idx : 0u));
                s_fc2[j] = s.fc2;
                split |= (s.col.w <= 1e30f);
            }
            const int any_split = __syncthreads_or(split);
            // back to front, 32 entries at a time: each lane tests one entry against the warp's pixels
            // and the warp walks those that can reach them and that one of its pixels reached in the forward pass
            for (int g = (cnt - 1) & ~31; g >= 0; g -= 32) {
                const int jl = g + lane;
                unsigned m = __ballot_sync(0xffffffffu, jl < cnt && lo + jl < wmax &&
                                                            meets_region(s_e[jl].pos, s_e[jl].con, s_e[jl].ext, reg));
                unsigned got = 0u;
                while (m) {
                    const int jb = 31 - __clz(m);
                    const unsigned bit = 1u << jb;
                    m ^= bit;
                    const int j = g + jb, e = lo + j;
                    // sums over this thread's pixels of dp, dp t and dp t^2 (dp = dL/d power) and of
                    // dL/drgb; the conic, opacity and mean terms are linear in these and in dy times them,
                    // so the warp reduces them and the CTA pass after the batch forms the terms
                    float S0 = 0.f, S1 = 0.f, S2 = 0.f, V0 = 0.f, V1 = 0.f, V2 = 0.f;
                    float wlast = 0.f;  // weight of the last pixel that blends the entry
                    const float4 P = s_e[j].pos;
                    const float4 K = s_e[j].con;
                    const float4 c = s_e[j].col;
                    const float dy = __fsub_rn(__fsub_rn(fj, P.y), P.w);
                    float centre, rowt;
                    row_terms(K, P.z, dy, centre, rowt);
                    float tk[PPT], pk[PPT];
                    if (!any_split) {
#pragma unroll
                        for (int k = 0; k < PPT; ++k) {
                            tk[k] = __fsub_rn(__fsub_rn(fik[k], P.x), centre);
                            pk[k] = slice_exponent(K, tk[k], rowt);
                        }
                    } else {
                        const float fc2 = s_fc2[j];
#pragma unroll
                        for (int k = 0; k < PPT; ++k) {
                            tk[k] = __fsub_rn(__fsub_rn(fik[k], fik[k] >= c.w ? fc2 : P.x), centre);
                            pk[k] = slice_exponent(K, tk[k], rowt);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < PPT; ++k) {
                        if (e >= nl[k] || !(pk[k] >= kLog2AlphaMin)) continue;
                        const float t = tk[k];
                        const float ar = alpha_exp2(pk[k]);
                        const float alpha = fminf(kAlphaMax, ar);
                        const float inv = rcp_approx(__fsub_rn(1.f, alpha));
                        const float Tj = T[k] * inv;
                        const float w = alpha * Tj;
                        wlast = w;
                        const float cg = c.x * g0[k] + c.y * g1[k] + c.z * g2[k];
                        V0 = fmaf(w, g0[k], V0);
                        V1 = fmaf(w, g1[k], V1);
                        V2 = fmaf(w, g2[k], V2);
                        const float dLda = Tj * cg - Bg[k] * inv;
                        Bg[k] = fmaf(cg, w, Bg[k]);
                        T[k] = Tj;
                        if (ar < kAlphaMax) {  // no gradient through the 0.99 clamp
                            const float dp = dLda * alpha;  // dL/d(power), power = ln G
                            const float dpt = dp * t;
                            S0 += dp;
                            S1 += dpt;
                            S2 = fmaf(dpt, t, S2);
                        }
                    }
                    if (!__any_sync(0xffffffffu, wlast > 0.f)) continue;  // no pixel blended the entry
                    got |= bit;
                    float* red = s_red + ((size_t)j * nwarps + warp) * 9;
                    // sum dp, sum dp t, sum dp t^2, sum dp t dy, sum dp dy, sum dp dy^2, dL/drgb
                    if (ROWS4) {
                        const float sm = warp_reduce_rows4(S0, S1, S2, V0, V1, V2, dy, lane);
                        if (slot4 >= 0) red[slot4] = sm;
                    } else {
                        const float dyS0 = dy * S0;
                        const float vals[9] = {S0, S1, S2, dy * S1, dyS0, dy * dyS0, V0, V1, V2};
                        int vi;
                        bool ok;
                        const float sm = warp_reduce9(vals, lane, &vi, &ok);
                        if (ok) red[vi] = sm;
                    }
                }
                if (lane == 0) s_got[2 * warp + (g >> 5)] = got;
            }
            __syncthreads();
            // per entry: the warps' sums added, then the screen-space gradient terms. With (dx, dy) =
            // pixel - mean and power = ln o - (a t^2 + gamma dy^2) / 2, t = dx - beta dy (the conic in
            // slice form), the gradients w.r.t. the mean, the slice-form conic and the opacity are
            //   dL/du = a sum(dp t), dL/dv = -a beta sum(dp t) + gamma sum(dp dy),
            //   dL/da = -sum(dp t^2) / 2, dL/dbeta = a sum(dp t dy), dL/dgamma = -sum(dp dy^2) / 2,
            //   dL/do = sum(dp) / o.
            // Each sum is dominated by its own scale (t across the ellipse, dy along it), so even for a
            // needle-like Gaussian the thin direction's information is not a small difference of the
            // long direction's sums, as the conic's image-axis entries would make it.
            for (int jj = tid; jj < cnt; jj += nthr) {
                float q[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) q[k] = 0.f;
                bool some = false;
                for (int w = 0; w < nwarps; ++w) {
                    if (!((s_got[2 * w + (jj >> 5)] >> (jj & 31)) & 1u)) continue;
                    some = true;
                    const float* r = s_red + ((size_t)jj * nwarps + w) * 9;
#pragma unroll
                    for (int k = 0; k < 9; ++k) q[k] += r[k];
                }
                if (!some) continue;
                const float4 R = s_e[jj].raw;  // a, gamma, 1 / o, item
                const float du_ = R.x * q[1];
                const float4 p0 = make_float4(du_, fmaf(R.y, q[4], -s_e[jj].con.y * du_), -0.5f * q[2], R.x * q[3]);
                const float4 p1 = make_float4(-0.5f * q[5], R.z * q[0], q[6], q[7]);
                float4* dst = a.acc + 3 * (size_t)__float_as_uint(R.w);
                if (p0.x != 0.f || p0.y != 0.f || p0.z != 0.f || p0.w != 0.f) red_add_v4(dst, p0);
                if (p1.x != 0.f || p1.y != 0.f || p1.z != 0.f || p1.w != 0.f) red_add_v4(dst + 1, p1);
                if (q[8] != 0.f) red_add_v4(dst + 2, make_float4(q[8], 0.f, 0.f, 0.f));
            }
            __syncthreads();  // the next batch overwrites the staged entries and s_red
        }
    }
    unsigned long long ev = evals;
    for (int o = 16; o > 0; o >>= 1) ev += __shfl_xor_sync(0xffffffffu, ev, o);
    if (lane == 0 && ev) atomicAdd(&a.hdr->evals_bwd, ev);
}

size_t render_bwd_smem(int batch, int threads) {
    return (size_t)batch * (sizeof(StagedBwd) + sizeof(float)) + (size_t)batch * (threads / 32) * 9 * sizeof(float) +
           (size_t)(threads / 32) * 2 * sizeof(uint32_t);
}

namespace {

using BwdKernel = void (*)(BwdArgs);

// The kernel for a tile and pixels per thread: four lanes per pixel row have their own reduction.
BwdKernel bwd_kernel(int tile_w, int tile_h, int ppt) {
    const bool rows4 = region_width(tile_w, tile_h, ppt) == 4 * ppt;
    switch (ppt) {
        case 8: return rows4 ? k_render_bwd<8, true> : k_render_bwd<8, false>;
        case 4: return rows4 ? k_render_bwd<4, true> : k_render_bwd<4, false>;
        case 2: return rows4 ? k_render_bwd<2, true> : k_render_bwd<2, false>;
        case 1: return rows4 ? k_render_bwd<1, true> : k_render_bwd<1, false>;
    }
    return nullptr;
}

}  // namespace

int render_bwd_occupancy(int tile_w, int tile_h, int batch, int ppt) {
    const BwdKernel k = bwd_kernel(tile_w, tile_h, ppt);
    if (!k) return 1;
    const int threads = tile_w * tile_h / ppt;
    int nb = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, threads, render_bwd_smem(batch, threads));
    return (e == cudaSuccess && nb > 0) ? nb : 1;
}

cudaError_t launch_render_bwd(const BwdArgs& a, int grid, cudaStream_t st) {
    const BwdKernel k = bwd_kernel(a.tile_w, a.tile_h, a.ppt);
    if (!k) return cudaErrorInvalidValue;
    const int threads = a.tile_w * a.tile_h / a.ppt;
    k<<<grid, threads, render_bwd_smem(a.batch, threads), st>>>(a);
    return cudaGetLastError();
}

}  // namespace odgs
