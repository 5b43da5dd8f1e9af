// L1 + D-SSIM loss of 3DGS training on ERP images, forward and gradient (sm_103a).
//
// SSIM_mean = sum_q c_q s_q with c_q the pixel's weight (cos(theta) of its row, or 1) over the
// weight of all 3 W H values, and s_q = (2 mx my + C1)(2 sxy + C2) / ((mx^2 + my^2 + C1)(sxx + syy + C2))
// from window moments mx = g * x, sxx = g * x^2 - mx^2, sxy = g * xy - mx my (g: the separable
// 11-tap Gaussian). Because every moment is a correlation with g, which is symmetric,
//   dSSIM_mean / dx_p = (g * A)_p + 2 x_p (g * B)_p + y_p (g * C)_p,
//   A = c (ds/dmx - 2 mx ds/dsxx - my ds/dsxy),  B = c ds/dsxx,  C = c ds/dsxy.
//   k_ssim_fwd    a warp streams down a strip of 64 columns (two per lane): per row the horizontal
//                 11-tap sums of the five moments from a row buffer in shared memory (a ring of eight
//                 rows filled by cp.async), then the vertical sums as a FIR filter in transposed form
//                 in registers (ten pending sums per moment and column), so that each finished row
//                 gives s, the loss partial and the maps A, B, C (scratch) with no second pass
//                 over shared memory and no barrier but the warp's
//   k_ssim_bwd    the same over A, B, C, then the gradient with the L1 term
// Measured at 2048 x 1024 against 32 x 32 tiles with both passes in shared memory: 104 -> 56 us and
// 121 -> 43 us. The rows in registers instead of the ring, one ahead: 74 and 82 us.
//   k_l1          lambda = 0: the L1 term alone, one pass
//   k_loss_reduce one CTA: the CTAs' partials in a fixed order (deterministic)
// Rows outside the image are zero (zero padding); columns wrap around the seam or are zero.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>

#include "odgs_train.h"

namespace {

constexpr int kR = 5;
constexpr int kWin = 2 * kR + 1;
constexpr int kTaps = 2 * kR;   // pending vertical sums per moment and column
constexpr int kCols = 64;       // columns of a warp's strip
constexpr int kRow = kCols + 2 * kR + 2;  // row buffer, padded to whole 16-byte reads
constexpr int kRing = 8;        // rows in flight per warp: a row takes an SM less time than a load
constexpr int kThreads = 256;
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

struct LossArgs {
    const float* x;
    const float* y;
    float* grad;
    float2* ab;      // maps A, B: [3 channels][H][pitch]
    float* c;        // map C: [3 channels][H][pitch]
    float* partial;  // [CTAs]
    int W, H, wrap, area;
    int pitch;                // row stride of the maps: W rounded up to whole 16-byte groups
    int strips, segs, rows;   // strips of kCols columns, segments of `rows` rows
    float lam, inv_wsum;
    float g[kWin];
};

__device__ __forceinline__ float row_weight(const LossArgs& a, int j) {
    // cos of the row centre's elevation pi (1/2 - (j + 1/2) / H) = sin(pi (j + 1/2) / H)
    return a.area ? sinpif(((float)j + 0.5f) / (float)a.H) : 1.f;
}

// Two single-precision operations in one instruction, each half rounded as the scalar one. The window
// sums of (x, y), of (x^2, y^2) and of the maps (A, B) run in pairs.
__device__ __forceinline__ unsigned long long pack2(float2 v) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
    return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}

// Asynchronous copies into shared memory, zero-filled where !ok.
__device__ __forceinline__ void copy4(float* dst, const float* src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void copy8(float2* dst, const float2* src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// One row's horizontal sum h enters the vertical filter; returns the finished sum, of the row kR rows
// earlier (transposed form: each pending sum takes its tap of h and moves down by one).
__device__ __forceinline__ float2 fir_step(float2 (&acc)[kTaps], float2 h, const float* g) {
    const float2 out = fma2(make_float2(g[0], g[0]), h, acc[0]);
#pragma unroll
    for (int i = 0; i < kTaps - 1; ++i) acc[i] = fma2(make_float2(g[i + 1], g[i + 1]), h, acc[i + 1]);
    acc[kTaps - 1] = mul2(make_float2(g[kTaps], g[kTaps]), h);
    return out;
}
__device__ __forceinline__ float fir_step(float (&acc)[kTaps], float h, const float* g) {
    const float out = fmaf(g[0], h, acc[0]);
#pragma unroll
    for (int i = 0; i < kTaps - 1; ++i) acc[i] = fmaf(g[i + 1], h, acc[i + 1]);
    acc[kTaps - 1] = g[kTaps] * h;
    return out;
}

// The strip, segment and channel of a warp (one per CTA), and the columns its lanes load: lane + 32 q
// from the strip's first less kR, wrapped or -1 (zero) outside the image.
struct Strip {
    int x0, y0, y1, ch;
    int col[3];
};
__device__ __forceinline__ Strip make_strip(const LossArgs& a, int lane) {
    Strip s;
    int k = blockIdx.x;
    s.x0 = (k % a.strips) * kCols;
    k /= a.strips;
    s.y0 = (k % a.segs) * a.rows;
    s.ch = k / a.segs;
    s.y1 = min(s.y0 + a.rows, a.H);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        int x = s.x0 - kR + lane + 32 * q;
        if (a.wrap) {
            x = ((x % a.W) + a.W) % a.W;
        } else if (x < 0 || x >= a.W) {
            x = -1;
        }
        s.col[q] = lane + 32 * q < kCols + 2 * kR ? x : -1;
    }
    return s;
}

__device__ __forceinline__ float block_sum(float v, float* s_red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < kThreads / 32; ++w) t += s_red[w];
    return t;
}

// Forward: loss partials and the maps A, B, C. 11 taps x 5 moments x 2 passes per value; a lane's two
// columns share the row buffer's reads and the products.
__global__ void __launch_bounds__(32) k_ssim_fwd(LossArgs a) {
    __shared__ __align__(16) float2 s_row[kRing][kRow];
    const int lane = threadIdx.x;
    const Strip st = make_strip(a, lane);
    const size_t HW = (size_t)a.W * a.H;
    const float* __restrict__ px = a.x + st.ch * HW;
    const float* __restrict__ py = a.y + st.ch * HW;
    float2 m1[2][kTaps], m2[2][kTaps];  // pending sums of (x, y) and (x^2, y^2)
    float m3[2][kTaps];                 // of xy
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < kTaps; ++i) {
            m1[j][i] = m2[j][i] = make_float2(0.f, 0.f);
            m3[j][i] = 0.f;
        }
    const int gx = st.x0 + 2 * lane;
    const int r0 = max(st.y0 - kR, 0), rend = st.y1 + kR;
    auto fetch = [&](int r) {  // row r, interleaved (x, y)
        float2* row = s_row[r % kRing];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (32 * q + lane >= kRow) continue;
            const bool ok = st.col[q] >= 0 && r < a.H && r < rend;
            const size_t o = ok ? (size_t)r * a.W + st.col[q] : 0;
            copy4(&row[32 * q + lane].x, px + o, ok);
            copy4(&row[32 * q + lane].y, py + o, ok);
        }
        copy_commit();
    };
    for (int k = 0; k < kRing - 1; ++k) fetch(r0 + k);
    float part = 0.f, wv = 0.f, wo = 0.f;  // row weights of 32 loaded and of 32 finished rows
    for (int r = r0; r < rend; ++r) {
        const float2* row = s_row[r % kRing];
        copy_wait<kRing - 2>();
        __syncwarp();  // row r is in place, and every lane is done with the row the next copy replaces
        fetch(r + kRing - 1);
        // horizontal sums of columns gx and gx + 1: 12 inputs
        float2 h1[2], h2[2];
        float h3[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            h1[j] = h2[j] = make_float2(0.f, 0.f);
            h3[j] = 0.f;
        }
        float2 centre[2];
#pragma unroll
        for (int i = 0; i < kWin + 1; i += 2) {
            const float4 v4 = *reinterpret_cast<const float4*>(row + 2 * lane + i);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float2 v = e ? make_float2(v4.z, v4.w) : make_float2(v4.x, v4.y);
                const float2 vv = mul2(v, v);
                const float xy = v.x * v.y;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int k = i + e - j;
                    if (k < 0 || k >= kWin) continue;
                    const float2 gk = make_float2(a.g[k], a.g[k]);
                    h1[j] = fma2(gk, v, h1[j]);
                    h2[j] = fma2(gk, vv, h2[j]);
                    h3[j] = fmaf(a.g[k], xy, h3[j]);
                    if (k == kR) centre[j] = v;
                }
            }
        }
        if (r >= st.y0 && r < st.y1) {  // the L1 term of this row
            if (((r - st.y0) & 31) == 0) wv = row_weight(a, r + lane);
            const float w = __shfl_sync(0xffffffffu, wv, (r - st.y0) & 31);
            float d = 0.f;
#pragma unroll
            for (int j = 0; j < 2; ++j) d += gx + j < a.W ? fabsf(centre[j].x - centre[j].y) : 0.f;
            part = fmaf(w * a.inv_wsum * (1.f - a.lam), d, part);
        }
        const int y = r - kR;
        const bool done = y >= st.y0;  // warp-uniform
        if (done && ((y - st.y0) & 31) == 0) wo = row_weight(a, y + lane);
        const float w = __shfl_sync(0xffffffffu, wo, (y - st.y0) & 31) * a.inv_wsum;
        float oa[2], ob[2], oc[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 m = fir_step(m1[j], h1[j], a.g), s = fir_step(m2[j], h2[j], a.g);
            const float e = fir_step(m3[j], h3[j], a.g);
            const float mx = m.x, my = m.y;
            const float sxx = s.x - mx * mx, syy = s.y - my * my, sxy = e - mx * my;
            const float A1 = 2.f * mx * my + kC1, A2 = 2.f * sxy + kC2;
            const float B1 = mx * mx + my * my + kC1, B2 = sxx + syy + kC2;
            const float iB = 1.f / (B1 * B2), iB1 = B2 * iB, iB2 = B1 * iB;
            const float sv = A1 * A2 * iB;
            const float ds_dmx = 2.f * A2 * (my * B1 - mx * A1) * iB1 * iB;
            const float ds_dsxx = -sv * iB2;
            const float ds_dsxy = 2.f * A1 * iB;
            if (done && gx + j < a.W) part = fmaf(w * a.lam, 1.f - sv, part);
            oa[j] = w * (ds_dmx - 2.f * mx * ds_dsxx - my * ds_dsxy);
            ob[j] = w * ds_dsxx;
            oc[j] = w * ds_dsxy;
        }
        if (done && gx < a.W) {  // the pitch leaves room for a last odd column's pair
            const size_t o = ((size_t)st.ch * a.H + y) * a.pitch + gx;
            *reinterpret_cast<float4*>(a.ab + o) = make_float4(oa[0], ob[0], oa[1], ob[1]);
            *reinterpret_cast<float2*>(a.c + o) = make_float2(oc[0], oc[1]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) a.partial[blockIdx.x] = part;
}

// Backward: the same streaming sums over the maps A, B, C, then the gradient with the L1 term.
__global__ void __launch_bounds__(32) k_ssim_bwd(LossArgs a) {
    __shared__ __align__(16) float2 s_row[kRing][kRow];
    __shared__ __align__(16) float s_c[kRing][kRow];
    __shared__ __align__(16) float s_x[kRing][kCols], s_y[kRing][kCols];  // the image rows being finished
    const int lane = threadIdx.x;
    const Strip st = make_strip(a, lane);
    const size_t HW = (size_t)a.W * a.H;
    const float2* __restrict__ pab = a.ab + (size_t)st.ch * a.H * a.pitch;
    const float* __restrict__ pc = a.c + (size_t)st.ch * a.H * a.pitch;
    const float* __restrict__ px = a.x + st.ch * HW;
    const float* __restrict__ py = a.y + st.ch * HW;
    float2 m1[2][kTaps];
    float m3[2][kTaps];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int i = 0; i < kTaps; ++i) {
            m1[j][i] = make_float2(0.f, 0.f);
            m3[j][i] = 0.f;
        }
    const int gx = st.x0 + 2 * lane;
    const int r0 = max(st.y0 - kR, 0), rend = st.y1 + kR;
    const bool in0 = gx < a.W, in1 = gx + 1 < a.W;
    const bool pair = in1 && (a.W & 1) == 0 && (reinterpret_cast<uintptr_t>(a.grad) & 7u) == 0;
    auto fetch = [&](int r) {  // row r of the maps, row r - kR of the images
        float2* row = s_row[r % kRing];
        float* rowc = s_c[r % kRing];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            if (32 * q + lane >= kRow) continue;
            const bool ok = st.col[q] >= 0 && r < a.H && r < rend;
            const size_t o = ok ? (size_t)r * a.pitch + st.col[q] : 0;
            copy8(row + 32 * q + lane, pab + o, ok);
            copy4(rowc + 32 * q + lane, pc + o, ok);
        }
        const int y = r - kR;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int x = st.x0 + 32 * q + lane;
            const bool ok = y >= st.y0 && y < st.y1 && x < a.W;
            const size_t o = ok ? (size_t)y * a.W + x : 0;
            copy4(&s_x[r % kRing][32 * q + lane], px + o, ok);
            copy4(&s_y[r % kRing][32 * q + lane], py + o, ok);
        }
        copy_commit();
    };
    for (int k = 0; k < kRing - 1; ++k) fetch(r0 + k);
    float wo = 0.f;
    for (int r = r0; r < rend; ++r) {
        const float2* row = s_row[r % kRing];
        const float* rowc = s_c[r % kRing];
        copy_wait<kRing - 2>();
        __syncwarp();  // row r is in place, and every lane is done with the row the next copy replaces
        fetch(r + kRing - 1);
        const int y = r - kR;
        const bool done = y >= st.y0;  // warp-uniform
        const size_t pix = (size_t)st.ch * HW + (size_t)y * a.W + gx;
        const float2 xv2 = *reinterpret_cast<const float2*>(&s_x[r % kRing][2 * lane]);
        const float2 yv2 = *reinterpret_cast<const float2*>(&s_y[r % kRing][2 * lane]);
        const float xv[2] = {xv2.x, xv2.y}, yv[2] = {yv2.x, yv2.y};
        float2 h1[2];
        float h3[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            h1[j] = make_float2(0.f, 0.f);
            h3[j] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kWin + 1; i += 2) {
            const float4 v4 = *reinterpret_cast<const float4*>(row + 2 * lane + i);
            const float2 c2 = *reinterpret_cast<const float2*>(rowc + 2 * lane + i);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float2 v = e ? make_float2(v4.z, v4.w) : make_float2(v4.x, v4.y);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int k = i + e - j;
                    if (k < 0 || k >= kWin) continue;
                    h1[j] = fma2(make_float2(a.g[k], a.g[k]), v, h1[j]);
                    h3[j] = fmaf(a.g[k], e ? c2.y : c2.x, h3[j]);
                }
            }
        }
        if (done && ((y - st.y0) & 31) == 0) wo = row_weight(a, y + lane);
        const float w = __shfl_sync(0xffffffffu, wo, (y - st.y0) & 31) * a.inv_wsum;
        float gr[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 m = fir_step(m1[j], h1[j], a.g);
            const float e = fir_step(m3[j], h3[j], a.g);
            const float d = xv[j] - yv[j];
            const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
            gr[j] = (1.f - a.lam) * w * sgn - a.lam * (m.x + 2.f * xv[j] * m.y + yv[j] * e);
        }
        if (done) {
            if (pair) {
                *reinterpret_cast<float2*>(a.grad + pix) = make_float2(gr[0], gr[1]);
            } else {
                if (in0) a.grad[pix] = gr[0];
                if (in1) a.grad[pix + 1] = gr[1];
            }
        }
    }
}

// The L1 term alone (lambda = 0) of up to kL1Views views in one launch, a (view, channel, row) per step
// of a CTA: the weighted |x - y| and the gradient w sign(x - y) / (weight sum), one pass over the pixels
// at the copy bandwidth. A launch and a reduction per view took 180 us for the 16 views of three sizes
// whose 700 MB take 103 us. Up to 8192 CTAs, mostly one per step: a CTA's loads end with its row, so the next row's
// have to be another CTA's. With as many as are resident (1216), each taking several rows, 16384 x 4096
// takes 379 us instead of 350 (2432: 365; 4864: 354), 8 views of 4096 x 2048 376 instead of 350 and one 53.8 instead of 51.4.
// Frames of few or narrow rows take 1216: a CTA per row of six views of 208 x 208 costs it and the reduction 13.7 -> 16.4 us.
constexpr int kL1Views = 64;
struct L1View {
    const float* x;
    const float* y;
    float* grad;
    int W, H, area;
    float inv_wsum;
    int row0;  // first of its 3 H rows
};
struct L1Args {
    L1View v[kL1Views];
    int views, rows;
    float* partial;  // [CTAs]
};

__global__ void __launch_bounds__(kThreads) k_l1(const __grid_constant__ L1Args a) {
    __shared__ float s_red[kThreads / 32];
    float part = 0.f;
    int k = 0;
    for (int rc = blockIdx.x; rc < a.rows; rc += gridDim.x) {
        while (k + 1 < a.views && rc >= a.v[k + 1].row0) ++k;
        const L1View& V = a.v[k];
        const int row = (rc - V.row0) % V.H;
        // cos of the row centre's elevation, as row_weight
        const float w = (V.area ? sinpif(((float)row + 0.5f) / (float)V.H) : 1.f) * V.inv_wsum;
        const size_t base = (size_t)(rc - V.row0) * V.W;
        const float* __restrict__ x = V.x + base;
        const float* __restrict__ y = V.y + base;
        float* __restrict__ g = V.grad ? V.grad + base : nullptr;
        // 16-byte loads and stores when every row starts on a 16-byte boundary
        const bool vec = (V.W & 3) == 0 && ((reinterpret_cast<uintptr_t>(V.x) | reinterpret_cast<uintptr_t>(V.y) |
                                             reinterpret_cast<uintptr_t>(V.grad)) & 15u) == 0;
        if (vec) {
            for (int c4 = threadIdx.x; c4 < (V.W >> 2); c4 += kThreads) {
                const float4 xv = __ldg(reinterpret_cast<const float4*>(x) + c4);
                const float4 yv = __ldg(reinterpret_cast<const float4*>(y) + c4);
                const float d[4] = {xv.x - yv.x, xv.y - yv.y, xv.z - yv.z, xv.w - yv.w};
                float gq[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    part = fmaf(w, fabsf(d[q]), part);
                    gq[q] = d[q] > 0.f ? w : (d[q] < 0.f ? -w : 0.f);
                }
                if (g) reinterpret_cast<float4*>(g)[c4] = make_float4(gq[0], gq[1], gq[2], gq[3]);
            }
            continue;
        }
        for (int col = threadIdx.x; col < V.W; col += kThreads) {
            const float d = x[col] - y[col];
            part = fmaf(w, fabsf(d), part);
            if (g) g[col] = d > 0.f ? w : (d < 0.f ? -w : 0.f);
        }
    }
    const float t = block_sum(part, s_red);
    if (threadIdx.x == 0) a.partial[blockIdx.x] = t;
}

__global__ void __launch_bounds__(kThreads) k_loss_reduce(const float* __restrict__ partial, int n, float* loss,
                                                          int accumulate) {
    __shared__ float s_red[kThreads / 32];
    float v = 0.f;
    for (int i = threadIdx.x; i < n; i += kThreads) v += partial[i];
    const float t = block_sum(v, s_red);
    if (threadIdx.x == 0) *loss = accumulate ? *loss + t : t;
}

constexpr int kSms = 152;  // GB300
constexpr int kL1Blocks = 8192, kL1Few = 8 * kSms;  // CTAs of the L1 pass alone, as far as the scratch holds their sums
constexpr int kL1Values = 2048;                     // it is worth one for

// 1 over the sum of an image's pixel weights; the sum over j of sin(pi (j + 1/2) / H) is 1 / sin(pi / (2 H))
float inv_weight_sum(int W, int H, int area) {
    return (float)(1.0 / (3.0 * W * (area ? 1.0 / std::sin(M_PI / (2.0 * H)) : (double)H)));
}

// Strips and segments of the streaming passes, one warp each. A segment reads 2 kR rows more than it
// finishes, and an SM needs about kBusy warps to hide the latencies: the number of segments that
// minimises the rows the fullest SM works through (at 2048 x 1024 with kBusy 8 / 12 / 16: 72 + 51,
// 56 + 43, 62 + 44 us).
struct Plan {
    int strips, segs, rows, pitch;
    int warps() const { return 3 * strips * segs; }
};
Plan make_plan(int W, int H) {
    constexpr int kBusy = 12;
    Plan p{};
    p.strips = (W + kCols - 1) / kCols;
    p.pitch = (W + 3) & ~3;
    long long best = -1;
    for (int segs = 1; segs <= (H + 7) / 8; ++segs) {
        const int rows = (H + segs - 1) / segs;
        const long long warps = 3ll * p.strips * ((H + rows - 1) / rows);
        const long long cost = std::max<long long>((warps + kSms - 1) / kSms, kBusy) * (rows + 2 * kR);
        if (best < 0 || cost < best) {
            best = cost;
            p.rows = rows;
            p.segs = (H + rows - 1) / rows;
        }
    }
    return p;
}

size_t maps_bytes(const Plan& p, int H) { return (9 * (size_t)p.pitch * H * sizeof(float) + 15) & ~(size_t)15; }
size_t scratch_for(int W, int H) {
    const Plan p = make_plan(W, H);
    return maps_bytes(p, H) + (size_t)std::max(p.warps(), kL1Few) * sizeof(float);
}

}  // namespace

extern "C" odgs_status odgs_loss_scratch_size(int width, int height, size_t* bytes) {
    if (!bytes || width < 1 || height < 1) return ODGS_ERR_INVALID_ARG;
    *bytes = scratch_for(width, height);
    return ODGS_OK;
}

extern "C" odgs_status odgs_loss_l1(const float* const* images, const float* const* targets, const int* widths,
                                    const int* heights, int n_views, const odgs_loss_params* p, float* const* grads,
                                    float* loss, void* scratch, size_t scratch_bytes, void* stream) {
    if (!images || !targets || !widths || !heights || n_views < 1 || !p || !loss) return ODGS_ERR_INVALID_ARG;
    for (int k = 0; k < n_views; ++k)
        if (!images[k] || !targets[k] || widths[k] < 1 || heights[k] < 1 || heights[k] > INT_MAX / 3)
            return ODGS_ERR_INVALID_ARG;
    if (!scratch || (reinterpret_cast<uintptr_t>(scratch) & 15u) || scratch_bytes < kL1Few * sizeof(float))
        return ODGS_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int most = (int)std::min<size_t>(kL1Blocks, scratch_bytes / sizeof(float));
    for (int k = 0; k < n_views;) {
        const bool first = k == 0;
        L1Args a{};
        a.partial = static_cast<float*>(scratch);
        long long values = 0;
        for (; k < n_views && a.views < kL1Views && (a.views == 0 || heights[k] <= (INT_MAX - a.rows) / 3); ++k) {
            L1View& v = a.v[a.views++];
            v.x = images[k];
            v.y = targets[k];
            v.grad = grads ? grads[k] : nullptr;
            v.W = widths[k];
            v.H = heights[k];
            v.area = p->area_weight ? 1 : 0;
            v.inv_wsum = inv_weight_sum(v.W, v.H, v.area);
            v.row0 = a.rows;
            a.rows += 3 * v.H;
            values += 3ll * v.W * v.H;
        }
        const int blocks = (int)std::min<long long>(a.rows, std::clamp<long long>(values / kL1Values, kL1Few, most));
        k_l1<<<blocks, kThreads, 0, st>>>(a);
        k_loss_reduce<<<1, kThreads, 0, st>>>(a.partial, blocks, loss, (p->accumulate || !first) ? 1 : 0);
    }
    return cudaGetLastError() == cudaSuccess ? ODGS_OK : ODGS_ERR_CUDA;
}

extern "C" odgs_status odgs_loss_l1_dssim(const float* image, const float* target, int width, int height,
                                          const odgs_loss_params* p, float* grad, float* loss, void* scratch,
                                          size_t scratch_bytes, void* stream) {
    if (!image || !target || !p || !loss || width < 1 || height < 1) return ODGS_ERR_INVALID_ARG;
    if (!(p->lambda >= 0.f && p->lambda <= 1.f)) return ODGS_ERR_INVALID_ARG;
    if (!scratch || (reinterpret_cast<uintptr_t>(scratch) & 15u) || scratch_bytes < scratch_for(width, height))
        return ODGS_ERR_WORKSPACE;
    if (p->lambda == 0.f)  // L1 alone: no SSIM window
        return odgs_loss_l1(&image, &target, &width, &height, 1, p, grad ? &grad : nullptr, loss, scratch, scratch_bytes,
                            stream);
    LossArgs a{};
    a.x = image; a.y = target; a.grad = grad;
    const Plan plan = make_plan(width, height);
    a.ab = static_cast<float2*>(scratch);
    a.c = reinterpret_cast<float*>(a.ab + 3 * (size_t)plan.pitch * height);
    a.partial = reinterpret_cast<float*>(static_cast<char*>(scratch) + maps_bytes(plan, height));
    a.W = width; a.H = height; a.wrap = p->wrap_u ? 1 : 0; a.area = p->area_weight ? 1 : 0;
    a.pitch = plan.pitch; a.strips = plan.strips; a.segs = plan.segs; a.rows = plan.rows;
    a.lam = p->lambda;
    a.inv_wsum = inv_weight_sum(width, height, a.area);
    double gsum = 0.0;
    double g[kWin];
    for (int k = 0; k < kWin; ++k) {
        const double d = k - kR;
        g[k] = std::exp(-d * d / (2.0 * 1.5 * 1.5));
        gsum += g[k];
    }
    for (int k = 0; k < kWin; ++k) a.g[k] = (float)(g[k] / gsum);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    k_ssim_fwd<<<plan.warps(), 32, 0, st>>>(a);
    k_loss_reduce<<<1, kThreads, 0, st>>>(a.partial, plan.warps(), loss, p->accumulate ? 1 : 0);
    if (grad) k_ssim_bwd<<<plan.warps(), 32, 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? ODGS_OK : ODGS_ERR_CUDA;
}
