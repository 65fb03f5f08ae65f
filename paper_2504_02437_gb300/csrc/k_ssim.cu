// The SSIM term of Eq. 10 (Section 3.2 "Map Optimization"):
//   L_color = (1 - lambda_photo) L1 + lambda_photo (1 - SSIM),
// SSIM averaged over the 3HW channel-pixels of a view, with the 3DGS
// lineage's window: an 11 x 11 Gaussian (sigma 1.5) normalised to sum 1,
// zero padding outside the image, C1 = 0.01^2, C2 = 0.03^2.
//
// Forward: per (plane, 32 x 32 tile) CTA, the rendered image x and the
// target y are staged with a 5-pixel halo; the five local moments (mu_x, mu_y,
// E[x^2], E[y^2], E[xy]) are blurred separably (rows, then columns), and each
// pixel q stores SSIM(q) and the three partial derivatives of SSIM(q) with
// respect to mu_x(q), E[x^2](q) and E[xy](q).
// Backward: dSSIM/dx(p) = sum_q w(q - p) [d/dmu_x + 2 x(p) d/dE[x^2]
// + y(p) d/dE[xy]](q): the three derivative maps are blurred the same way
// (the window is symmetric; pixels q outside the image do not exist, so the
// maps are zero-padded), and dL/dC combines it with the L1 sign term.
//
// Bound: 20 bytes in and out per channel-pixel forward, 24 backward, against some 90 multiply-adds;
// what a first version spent its time on was shared-memory loads, 22 and 55 a pixel in the two blurs.
// So a thread blurs four neighbouring outputs from the fourteen values they share, the quantities
// that are blurred alike sit side by side as pairs (x and y, x^2 and y^2, two of the derivative maps)
// and go through packed multiply-adds (each half rounds as the scalar operation does). Two views of
// 641x479: forward 40.6 -> 25 us, backward 43.8 -> 19 us.
#include <cmath>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kSsimTile = 32;
constexpr int kSsimRadius = 5;
constexpr int kSsimSpan = kSsimTile + 2 * kSsimRadius;   // 42
constexpr int kSsimThreads = 256;
constexpr float kSsimC1 = 0.01f * 0.01f, kSsimC2 = 0.03f * 0.03f;

struct SsimWindow {
    float w[2 * kSsimRadius + 1];
};

__device__ __forceinline__ float ssim_block_sum(float v, float* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x == 0)
        for (int k = 0; k < kSsimThreads / 32; ++k) t += sh[k];
    return t;   // valid in thread 0
}

// Two floats in one 64-bit register (the layout of a float2 in memory).
struct P2 {
    unsigned long long v;
};
__device__ __forceinline__ P2 p2_pack(float a, float b) {
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 p2_unpack(P2 x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x.v));
    return r;
}
__device__ __forceinline__ P2 p2_mul(P2 a, P2 b) {
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 p2_fma(P2 a, P2 b, P2 c) {
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

constexpr int kTaps = 2 * kSsimRadius + 1;
constexpr int kRun = 4, kShared = kRun + kTaps - 1;   // outputs a thread blurs together, values they share
// In the row blur a warp's lanes take the same columns of different rows: row lengths that are odd
// in 4-byte or 8-byte words keep them on different banks.
constexpr int kSpanPad = kSsimSpan + 1, kTilePad = kSsimTile + 1;

// Loads load(index of the pixel, or -1 outside the image) over the (kSsimSpan)^2 window around the
// tile, all of a thread's loads in flight at once, then store(r, c, value).
template <typename T, typename L, typename S>
__device__ __forceinline__ void stage_window(int W, int H, int x0, int y0, L load, S store) {
    constexpr int kN = (kSsimSpan * kSsimSpan + kSsimThreads - 1) / kSsimThreads;
    T v[kN];
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        const int i = threadIdx.x + u * kSsimThreads;
        const int r = i / kSsimSpan, cc = i - r * kSsimSpan;
        const int gx = x0 - kSsimRadius + cc, gy = y0 - kSsimRadius + r;
        v[u] = load(r < kSsimSpan && gx >= 0 && gx < W && gy >= 0 && gy < H ? (long)gy * W + gx : -1l);
    }
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        const int i = threadIdx.x + u * kSsimThreads;
        const int r = i / kSsimSpan, cc = i - r * kSsimSpan;
        if (r < kSsimSpan) store(r, cc, v[u]);
    }
}

__global__ void __launch_bounds__(kSsimThreads) k_ssim_fwd(const float* __restrict__ x, const float* __restrict__ y,
                                                           const float* const* __restrict__ y_slot, int W, int H,
                                                           SsimWindow win, float neg_scale, float constant,
                                                           float2* __restrict__ d_mu_xx, float* __restrict__ d_xy,
                                                           float* __restrict__ partials) {
    __shared__ __align__(16) P2 sxy[kSsimSpan][kSpanPad];
    __shared__ __align__(16) P2 hm[kSsimSpan][kTilePad], hq[kSsimSpan][kTilePad];   // x, y; x^2, y^2
    __shared__ __align__(16) float hxy[kSsimSpan][kTilePad];
    __shared__ float red[kSsimThreads / 32];
    if (y_slot != nullptr) y = *y_slot;   // a replayed graph's per-call target
    const int plane = blockIdx.z;
    const size_t HW = (size_t)W * H, off = (size_t)plane * HW;
    const int x0 = blockIdx.x * kSsimTile, y0 = blockIdx.y * kSsimTile;
    stage_window<float2>(
        W, H, x0, y0, [&](long o) { return o >= 0 ? make_float2(x[off + o], y[off + o]) : make_float2(0.f, 0.f); },
        [&](int r, int cc, float2 v) { sxy[r][cc] = p2_pack(v.x, v.y); });
    __syncthreads();
    // rows: blur along x for every staged row
    for (int i = threadIdx.x; i < kSsimSpan * (kSsimTile / kRun); i += kSsimThreads) {
        const int c0 = i / kSsimSpan * kRun, r = i - i / kSsimSpan * kSsimSpan;
        P2 m[kRun], q[kRun];
        float xy[kRun];
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            m[e] = q[e] = p2_pack(0.f, 0.f);
            xy[e] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kShared; ++k) {
            const P2 u = sxy[r][c0 + k], uu = p2_mul(u, u);
            const float2 v = p2_unpack(u);
            const float uv = v.x * v.y;
#pragma unroll
            for (int e = 0; e < kRun; ++e) {
                if (k < e || k - e >= kTaps) continue;
                const float wk = win.w[k - e];
                m[e] = p2_fma(p2_pack(wk, wk), u, m[e]);
                q[e] = p2_fma(p2_pack(wk, wk), uu, q[e]);
                xy[e] = fmaf(wk, uv, xy[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            hm[r][c0 + e] = m[e];
            hq[r][c0 + e] = q[e];
            hxy[r][c0 + e] = xy[e];
        }
    }
    __syncthreads();
    float acc = 0.f;
    {   // columns: four rows a thread
        const int cc = threadIdx.x & (kSsimTile - 1), r0 = (threadIdx.x / kSsimTile) * kRun;
        P2 m[kRun], q[kRun];
        float xy[kRun];
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            m[e] = q[e] = p2_pack(0.f, 0.f);
            xy[e] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kShared; ++k) {
            const P2 a = hm[r0 + k][cc], b = hq[r0 + k][cc];
            const float c = hxy[r0 + k][cc];
#pragma unroll
            for (int e = 0; e < kRun; ++e) {
                if (k < e || k - e >= kTaps) continue;
                const float wk = win.w[k - e];
                m[e] = p2_fma(p2_pack(wk, wk), a, m[e]);
                q[e] = p2_fma(p2_pack(wk, wk), b, q[e]);
                xy[e] = fmaf(wk, c, xy[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            const int gx = x0 + cc, gy = y0 + r0 + e;
            if (gx >= W || gy >= H) continue;
            const float2 mu = p2_unpack(m[e]), sq = p2_unpack(q[e]);
            const float mx = mu.x, my = mu.y;
            const float A = 2.f * mx * my + kSsimC1;
            const float B = 2.f * (xy[e] - mx * my) + kSsimC2;
            const float Cc = mx * mx + my * my + kSsimC1;
            const float D = (sq.x - mx * mx) + (sq.y - my * my) + kSsimC2;
            const float iden = 1.f / (Cc * D);
            const float s = A * B * iden;
            acc += s;
            // partial derivatives of s with respect to mu_x, E[x^2], E[xy]
            const float g_mu = (2.f * my * (B - A)) * iden - s * (2.f * mx * (D - Cc)) / (Cc * D);
            const float g_xx = -s / D;
            const float g_xy = 2.f * A * iden;
            const size_t o = off + (size_t)gy * W + gx;
            d_mu_xx[o] = make_float2(g_mu, g_xx);
            d_xy[o] = g_xy;
        }
    }
    const float t = ssim_block_sum(acc, red);
    if (threadIdx.x == 0) {
        const int bid = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        partials[bid] = t * neg_scale + (bid == 0 ? constant : 0.f);
    }
}

__global__ void __launch_bounds__(kSsimThreads) k_ssim_bwd(const float* __restrict__ x, const float* __restrict__ y,
                                                           const float* const* __restrict__ y_slot, int W, int H,
                                                           SsimWindow win, const float2* __restrict__ d_mu_xx,
                                                           const float* __restrict__ d_xy, float l1_scale,
                                                           float ssim_scale, float* __restrict__ dLdC,
                                                           float* __restrict__ partials) {
    __shared__ __align__(16) P2 sg[kSsimSpan][kSpanPad];
    __shared__ __align__(16) float se[kSsimSpan][kSpanPad];
    __shared__ __align__(16) P2 hg[kSsimSpan][kTilePad];
    __shared__ __align__(16) float he[kSsimSpan][kTilePad];
    __shared__ float red[kSsimThreads / 32];
    if (y_slot != nullptr) y = *y_slot;
    const int plane = blockIdx.z;
    const size_t HW = (size_t)W * H, off = (size_t)plane * HW;
    const int x0 = blockIdx.x * kSsimTile, y0 = blockIdx.y * kSsimTile;
    stage_window<float3>(
        W, H, x0, y0,
        [&](long o) {
            const float2 g = o >= 0 ? d_mu_xx[off + o] : make_float2(0.f, 0.f);
            return make_float3(g.x, g.y, o >= 0 ? d_xy[off + o] : 0.f);
        },
        [&](int r, int cc, float3 v) {
            sg[r][cc] = p2_pack(v.x, v.y);
            se[r][cc] = v.z;
        });
    // the pixels' own values, loaded while the maps are blurred
    const int cc = threadIdx.x & (kSsimTile - 1), r0 = (threadIdx.x / kSsimTile) * kRun;
    float xp[kRun], yp[kRun];
#pragma unroll
    for (int e = 0; e < kRun; ++e) {
        const bool in = x0 + cc < W && y0 + r0 + e < H;
        const size_t o = off + (size_t)(y0 + r0 + e) * W + x0 + cc;
        xp[e] = in ? x[o] : 0.f;
        yp[e] = in ? y[o] : 0.f;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSsimSpan * (kSsimTile / kRun); i += kSsimThreads) {
        const int c0 = i / kSsimSpan * kRun, r = i - i / kSsimSpan * kSsimSpan;
        P2 g[kRun];
        float v[kRun];
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            g[e] = p2_pack(0.f, 0.f);
            v[e] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kShared; ++k) {
            const P2 u = sg[r][c0 + k];
            const float c = se[r][c0 + k];
#pragma unroll
            for (int e = 0; e < kRun; ++e) {
                if (k < e || k - e >= kTaps) continue;
                const float wk = win.w[k - e];
                g[e] = p2_fma(p2_pack(wk, wk), u, g[e]);
                v[e] = fmaf(wk, c, v[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            hg[r][c0 + e] = g[e];
            he[r][c0 + e] = v[e];
        }
    }
    __syncthreads();
    float acc = 0.f;
    {
        P2 g[kRun];
        float v[kRun];
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            g[e] = p2_pack(0.f, 0.f);
            v[e] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kShared; ++k) {
            const P2 u = hg[r0 + k][cc];
            const float c = he[r0 + k][cc];
#pragma unroll
            for (int e = 0; e < kRun; ++e) {
                if (k < e || k - e >= kTaps) continue;
                const float wk = win.w[k - e];
                g[e] = p2_fma(p2_pack(wk, wk), u, g[e]);
                v[e] = fmaf(wk, c, v[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < kRun; ++e) {
            const int gx = x0 + cc, gy = y0 + r0 + e;
            if (gx >= W || gy >= H) continue;
            const float2 ab = p2_unpack(g[e]);
            const size_t o = off + (size_t)gy * W + gx;
            const float dS = ab.x + 2.f * xp[e] * ab.y + yp[e] * v[e];
            const float res = xp[e] - yp[e];
            acc += fabsf(res);
            dLdC[o] = l1_scale * (float)((res > 0.f) - (res < 0.f)) - ssim_scale * dS;
        }
    }
    const float t = ssim_block_sum(acc, red);
    if (threadIdx.x == 0) partials[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t * l1_scale;
}
static_assert(kSsimThreads == kSsimTile * (kSsimTile / kRun), "one run of rows a thread");

SsimWindow make_window() {
    SsimWindow win;
    double g[2 * kSsimRadius + 1], s = 0.0;
    for (int k = 0; k <= 2 * kSsimRadius; ++k) {
        const double d = k - kSsimRadius;
        g[k] = std::exp(-d * d / (2.0 * 1.5 * 1.5));
        s += g[k];
    }
    for (int k = 0; k <= 2 * kSsimRadius; ++k) win.w[k] = (float)(g[k] / s);
    return win;
}

}  // namespace

int ssim_blocks(int width, int height, int n_views) {
    return n_views * 3 * ((width + kSsimTile - 1) / kSsimTile) * ((height + kSsimTile - 1) / kSsimTile);
}

// L_color with the SSIM term for the rendered views: writes dL/dC and, into
// `partials` (2 ssim_blocks entries), the photometric loss as per-CTA terms.
cudaError_t launch_ssim_loss(gs_ctx* c, const DevConst& k, const float* rgb, const float* target,
                             const float* const* target_slot, float* partials, cudaStream_t s) {
    const int W = c->width, H = c->height, V = c->n_views;
    const float lp = c->cfg.lambda_photo;
    const float inv = 1.f / (float)(3 * (size_t)W * H);
    const float l1_scale = k.lambda_color * (1.f - lp) * inv, ssim_scale = k.lambda_color * lp * inv;
    const size_t HW = (size_t)W * H * 3 * V;
    float2* d_mu_xx = reinterpret_cast<float2*>(c->ssim_maps);   // two maps side by side, then the third
    float* d_xy = c->ssim_maps + 2 * HW;
    const dim3 grid((W + kSsimTile - 1) / kSsimTile, (H + kSsimTile - 1) / kSsimTile, 3 * V);
    const int nb = ssim_blocks(W, H, V);
    const SsimWindow win = make_window();
    c->launches += 2;
    k_ssim_fwd<<<grid, kSsimThreads, 0, s>>>(rgb, target, target_slot, W, H, win, -ssim_scale, k.lambda_color * lp * (float)V,
                                             d_mu_xx, d_xy, partials);
    k_ssim_bwd<<<grid, kSsimThreads, 0, s>>>(rgb, target, target_slot, W, H, win, d_mu_xx, d_xy, l1_scale, ssim_scale,
                                             c->dLdC, partials + nb);
    return cudaGetLastError();
}

}  // namespace gs
