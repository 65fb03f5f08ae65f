// Per-Gaussian projection (Eq. 1-2, Section 3.1) and its adjoint.
//
// One thread per (view, Gaussian). Parameters are read from the planar SoA
// [14][cap] (each row coalesced across a warp); outputs are a 48-byte raster
// record per (view, Gaussian), the depth key for the sort, and the number of
// tiles the pixel box touches.
#include "gs_internal.cuh"

namespace gs {
namespace {

// View-independent shape of one Gaussian (Eq. 1): scales and Sigma = R S S^T R^T.
struct Shape {
    float s[3];
    float S[6];            // Sigma (xx, xy, xz, yy, yz, zz)
};

// View-dependent projection (Eq. 2) of one Gaussian for one camera.
struct Proj {
    float tx, ty, tz;
    float xr, yr;          // x/z, y/z before clamping
    float xh, yh;          // clamped
    float J00, J02, J11, J12;
    float T0[3], T1[3];    // rows of J W
    float A, B, C, det;    // dilated 2D covariance
};

// Float-float ("double-float") arithmetic: a value is hi + lo with |lo| <=
// ulp(hi)/2, about 48 significant bits. Error-free transformations: TwoSum
// (Knuth, TAOCP vol. 2, 4.2.2) and TwoProduct through a fused multiply-add
// (Dekker 1971; with FMA as in Ogita, Rump and Oishi 2005). The intrinsics
// keep the compiler from contracting or reassociating the steps.
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ FF quick_two_sum(float a, float b) {   // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ FF ff_add(FF x, FF y) {
    const FF s = two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
// r0 m0 + r1 m1 + r2 m2 + t of float32 inputs
__device__ __forceinline__ FF ff_dot3_add(float r0, float m0, float r1, float m1, float r2, float m2, float t) {
    FF acc = two_prod(r0, m0);
    acc = ff_add(acc, two_prod(r1, m1));
    acc = ff_add(acc, two_prod(r2, m2));
    return ff_add(acc, FF{t, 0.f});
}
__device__ __forceinline__ FF ff_div(FF a, FF b) {
    const float q1 = __fdiv_rn(a.hi, b.hi);
    const FF p = two_prod(q1, b.hi);
    // remainder a - q1 b, to first order
    const float r = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p.hi), p.lo), __fsub_rn(a.lo, __fmul_rn(q1, b.lo)));
    return quick_two_sum(q1, __fdiv_rn(r, b.hi));
}
// f a + c
__device__ __forceinline__ FF ff_scale_add(FF a, float f, float c) {
    FF p = two_prod(a.hi, f);
    p = quick_two_sum(p.hi, __fmaf_rn(a.lo, f, p.lo));
    return ff_add(p, FF{c, 0.f});
}
// floor and fraction of hi + lo: returns the integer part, writes the fraction in [0, 1)
__device__ __forceinline__ float ff_floor_frac(FF a, float& frac) {
    float fl = floorf(a.hi);
    float f = __fadd_rn(__fsub_rn(a.hi, fl), a.lo);   // a.hi - fl is exact
    if (f < 0.f) {
        fl -= 1.f;
        f = __fadd_rn(f, 1.f);
    } else if (f >= 1.f) {
        fl += 1.f;
        f = __fsub_rn(f, 1.f);
    }
    frac = fminf(fmaxf(f, 0.f), 0x1.fffffep-1f);
    return fl;
}

__device__ __forceinline__ void load_params(const float* __restrict__ P, int cap, int i, float p[kParamRows]) {
#pragma unroll
    for (int r = 0; r < kParamRows; ++r) p[r] = __ldg(P + (size_t)r * cap + i);
}

// The normalised quaternion (w, x, y, z) and its rotation (row-major); returns the norm.
__device__ __forceinline__ float rotation_of(const float p[kParamRows], float q[4], float R[9]) {
    float qq = p[6] * p[6] + p[7] * p[7] + p[8] * p[8] + p[9] * p[9];
    const float qnorm = sqrtf(qq);
    float inv = 1.0f / qnorm;
    float w = p[6] * inv, x = p[7] * inv, y = p[8] * inv, z = p[9] * inv;
    q[0] = w; q[1] = x; q[2] = y; q[3] = z;
    R[0] = 1.f - 2.f * (y * y + z * z); R[1] = 2.f * (x * y - w * z);       R[2] = 2.f * (x * z + w * y);
    R[3] = 2.f * (x * y + w * z);       R[4] = 1.f - 2.f * (x * x + z * z); R[5] = 2.f * (y * z - w * x);
    R[6] = 2.f * (x * z - w * y);       R[7] = 2.f * (y * z + w * x);       R[8] = 1.f - 2.f * (x * x + y * y);
    return qnorm;
}

// Eq. 1 in float32.
__device__ __forceinline__ void shape_of(const float p[kParamRows], Shape& g) {
    g.s[0] = expf(p[3]);
    g.s[1] = expf(p[4]);
    g.s[2] = expf(p[5]);
    float q[4], R[9];
    rotation_of(p, q, R);
    float M[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) M[i * 3 + k] = R[i * 3 + k] * g.s[k];
    g.S[0] = M[0] * M[0] + M[1] * M[1] + M[2] * M[2];
    g.S[1] = M[0] * M[3] + M[1] * M[4] + M[2] * M[5];
    g.S[2] = M[0] * M[6] + M[1] * M[7] + M[2] * M[8];
    g.S[3] = M[3] * M[3] + M[4] * M[4] + M[5] * M[5];
    g.S[4] = M[3] * M[6] + M[4] * M[7] + M[5] * M[8];
    g.S[5] = M[6] * M[6] + M[7] * M[7] + M[8] * M[8];
}

// Eq. 2 in float32 for one camera: J at the clamped x/z, y/z; T = J W;
// Sigma2D = T Sigma T^T + dilation I.
__device__ __forceinline__ void project_one(const float p[kParamRows], const Shape& g, const DevCamera& cam,
                                            float dilation, Proj& o) {
    o.tx = cam.R[0] * p[0] + cam.R[1] * p[1] + cam.R[2] * p[2] + cam.t[0];
    o.ty = cam.R[3] * p[0] + cam.R[4] * p[1] + cam.R[5] * p[2] + cam.t[1];
    o.tz = cam.R[6] * p[0] + cam.R[7] * p[1] + cam.R[8] * p[2] + cam.t[2];
    float iz = 1.0f / o.tz;
    o.xr = o.tx * iz;
    o.yr = o.ty * iz;
    o.xh = fminf(fmaxf(o.xr, -cam.lim_x), cam.lim_x);
    o.yh = fminf(fmaxf(o.yr, -cam.lim_y), cam.lim_y);
    o.J00 = cam.fx * iz;
    o.J02 = -cam.fx * o.xh * iz;
    o.J11 = cam.fy * iz;
    o.J12 = -cam.fy * o.yh * iz;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o.T0[k] = o.J00 * cam.R[k] + o.J02 * cam.R[6 + k];
        o.T1[k] = o.J11 * cam.R[3 + k] + o.J12 * cam.R[6 + k];
    }
    float ST0[3], ST1[3];
    ST0[0] = g.S[0] * o.T0[0] + g.S[1] * o.T0[1] + g.S[2] * o.T0[2];
    ST0[1] = g.S[1] * o.T0[0] + g.S[3] * o.T0[1] + g.S[4] * o.T0[2];
    ST0[2] = g.S[2] * o.T0[0] + g.S[4] * o.T0[1] + g.S[5] * o.T0[2];
    ST1[0] = g.S[0] * o.T1[0] + g.S[1] * o.T1[1] + g.S[2] * o.T1[2];
    ST1[1] = g.S[1] * o.T1[0] + g.S[3] * o.T1[1] + g.S[4] * o.T1[2];
    ST1[2] = g.S[2] * o.T1[0] + g.S[4] * o.T1[1] + g.S[5] * o.T1[2];
    o.A = o.T0[0] * ST0[0] + o.T0[1] * ST0[1] + o.T0[2] * ST0[2] + dilation;
    o.B = o.T0[0] * ST1[0] + o.T0[1] * ST1[1] + o.T0[2] * ST1[2];
    o.C = o.T1[0] * ST1[0] + o.T1[1] * ST1[1] + o.T1[2] * ST1[2] + dilation;
    o.det = o.A * o.C - o.B * o.B;
}

// Projection of one (view, Gaussian) item; returns whether it is visible (has tiles).
__device__ __forceinline__ bool preprocess_one(const float* __restrict__ P, int n, int cap, int gid, int view,
                                               const DevCamera* __restrict__ cams, const DevConst& kc, int tile,
                                               float4* __restrict__ rec, uint32_t* __restrict__ tiles,
                                               uint32_t* __restrict__ dkey, float* __restrict__ depth, float& planar,
                                               uint32_t& key) {
    const DevCamera& cam = cams[view];
    size_t item = (size_t)view * n + gid;
    float p[kParamRows];
    load_params(P, cap, gid, p);
    Shape g;
    shape_of(p, g);
    // the Gaussian's planar term of Eq. 10: max(floor, smallest scale)
    planar = fmaxf(kc.reg_floor, fminf(g.s[0], fminf(g.s[1], g.s[2])));
    Proj o;
    project_one(p, g, cam, kc.dilation, o);
    // Screen mean and depth in float-float (the covariance stays float32): the
    // compositing subtracts u from pixel coordinates, and the rounding of u in
    // float32 (about 1e-4 px at 1000 px) would dominate the error of the
    // cancelling sums of the mean gradient.
    const FF tzf = ff_dot3_add(cam.R[6], p[0], cam.R[7], p[1], cam.R[8], p[2], cam.t[2]);
    const FF txf = ff_dot3_add(cam.R[0], p[0], cam.R[1], p[1], cam.R[2], p[2], cam.t[0]);
    const FF tyf = ff_dot3_add(cam.R[3], p[0], cam.R[4], p[1], cam.R[5], p[2], cam.t[1]);
    const float tz32 = tzf.hi;
    bool valid = (tzf.hi > kc.near_z || (tzf.hi == kc.near_z && tzf.lo > 0.f)) && (o.det > 0.f);
    const FF izx = ff_div(txf, tzf), izy = ff_div(tyf, tzf);
    const FF uf2 = ff_scale_add(izx, cam.fx, cam.cx), vf2 = ff_scale_add(izy, cam.fy, cam.cy);
    float idet = 1.0f / o.det;
    float ca = o.C * idet, cb = -o.B * idet, cc = o.A * idet;
    float mid = 0.5f * (o.A + o.C);
    float lam = mid + sqrtf(fmaxf(kc.lambda_floor, mid * mid - o.det));
    float r = ceilf(kc.radius_sigma * sqrtf(lam));
    // screen positions beyond +-2^23 px or radii beyond 2^22 px are culled
    valid = valid && fabsf(uf2.hi) < 8388608.f && fabsf(vf2.hi) < 8388608.f && r < 4194304.f;
    float ui = 0.f, uf = 0.f, vi = 0.f, vf = 0.f;
    uint32_t ntiles = 0;
    if (valid) {
        ui = ff_floor_frac(uf2, uf);
        vi = ff_floor_frac(vf2, vf);
        int x0, x1, y0, y1;
        if (pixel_box(ui, uf, vi, vf, r, cam.width, cam.height, x0, x1, y0, y1))
            ntiles = (uint32_t)((x1 / tile - x0 / tile + 1) * (y1 / tile - y0 / tile + 1));
        else
            valid = false;
    }
    float o_act = 1.0f / (1.0f + expf(-p[10]));
    // conic pre-scaled for exp2: power * log2(e) = a' dx^2 + b' dx dy + c' dy^2
    const float k1 = -0.5f * kLog2e, k2 = -kLog2e;
    rec[item * 3 + 0] = make_float4(ui, vi, valid ? r : -1.f, o_act);
    rec[item * 3 + 1] = make_float4(ca * k1, cb * k2, cc * k1, uf);
    rec[item * 3 + 2] = make_float4(p[11], p[12], p[13], vf);
    tiles[item] = ntiles;
    depth[item] = tz32;
    key = valid ? __float_as_uint(tz32) : 0xFFFFFFFFu;
    dkey[item] = key;
    return valid;
}

// One thread per (view, Gaussian) item; each CTA also writes how many of its 256
// consecutive items are visible (block_vis[view * gridDim.x + blockIdx.x]), the
// first step of the order-keeping compaction ahead of the depth sort, with the
// range of their keys, and the
// CTAs of view 0 the sum of their Gaussians' planar terms times reg_scale
// (reg_part[blockIdx.x]; the loss adds these partials in index order).
// Six CTAs of 256 threads per SM (at most 40 registers): 48 resident warps for a latency-bound
// per-thread chain (A/B on the 300k-Gaussian keyframe: iteration 0.5494 -> 0.5462 ms).
__global__ void __launch_bounds__(256, 6) k_preprocess(const float* __restrict__ P, int n, int cap,
                                                    const DevCamera* __restrict__ cams, DevConst kc, int tile,
                                                    float4* __restrict__ rec, uint32_t* __restrict__ tiles,
                                                    uint32_t* __restrict__ dkey,
                                                    float* __restrict__ depth, uint32_t* __restrict__ block_vis,
                                                    uint2* __restrict__ block_range,
                                                    float reg_scale, float* __restrict__ reg_part) {
    __shared__ float wsum[8];
    __shared__ uint2 wrange[8];
    const int gid = blockIdx.x * blockDim.x + threadIdx.x;
    const int view = blockIdx.y;
    bool vis = false;
    float planar = 0.f;
    uint32_t key = 0xFFFFFFFFu;
    if (gid < n) vis = preprocess_one(P, n, cap, gid, view, cams, kc, tile, rec, tiles, dkey, depth, planar, key);
    {
        const uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, key), hi = __reduce_max_sync(0xFFFFFFFFu, vis ? key : 0u);
        if ((threadIdx.x & 31) == 0) wrange[threadIdx.x >> 5] = make_uint2(lo, hi);
    }
    const int cnt = __syncthreads_count(vis);
    if (threadIdx.x == 0) {
        uint2 r = wrange[0];
        for (int w = 1; w < 8; ++w) r = make_uint2(umin(r.x, wrange[w].x), umax(r.y, wrange[w].y));
        block_vis[(size_t)view * gridDim.x + blockIdx.x] = (uint32_t)cnt;
        block_range[(size_t)view * gridDim.x + blockIdx.x] = r;
    }
    if (view == 0) {   // uniform over the CTA
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) planar += __shfl_xor_sync(0xFFFFFFFFu, planar, o);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = planar;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;
            for (int w = 0; w < 8; ++w) t += wsum[w];
            reg_part[blockIdx.x] = t * reg_scale;
        }
    }
}

// Order-keeping compaction of the visible items, in item order, so that equal depths keep
// ascending ids through the stable sort. CTA B takes the items of projection CTAs 4B .. 4B + 3
// (linear index view * gx + x): it first adds the visible counts of the projection CTAs before
// them (a few thousand values at most, read straight from block_vis: no separate scan launch),
// then writes each one's visible keys and items in turn; the last CTA writes the total and the
// range of the keys, and zeroes the pair total.
constexpr int kCompactSub = 4;
__global__ void __launch_bounds__(256) k_compact_visible(const uint32_t* __restrict__ kin, int n, int gx,
                                                         int nblocks, const uint32_t* __restrict__ block_vis,
                                                         const uint2* __restrict__ block_range,
                                                         uint32_t* __restrict__ kout, uint32_t* __restrict__ vout,
                                                         uint32_t* __restrict__ counts) {
    __shared__ uint32_t wsum[8];
    __shared__ uint32_t s_off;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int b0 = blockIdx.x * kCompactSub;
    {
        uint32_t pre = 0;
        for (int b = threadIdx.x; b < b0; b += 256) pre += block_vis[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(0xFFFFFFFFu, pre, o);
        if (lane == 0) wsum[w] = pre;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (int k = 0; k < 8; ++k) t += wsum[k];
            s_off = t;
        }
        __syncthreads();
    }
    uint32_t off = s_off;
    uint32_t lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    for (int j = 0; j < kCompactSub && b0 + j < nblocks; ++j) {
        const int b = b0 + j, view = b / gx, gid = (b - view * gx) * 256 + threadIdx.x;
        const size_t item = (size_t)view * n + gid;
        const uint32_t key = gid < n ? kin[item] : 0xFFFFFFFFu;
        const bool vis = key != 0xFFFFFFFFu;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, vis);
        __syncthreads();   // the previous sub-block's counts have been read
        if (lane == 0) wsum[w] = __popc(bal);
        __syncthreads();
        uint32_t pre = 0, cnt = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            pre += k < w ? wsum[k] : 0u;
            cnt += wsum[k];
        }
        if (vis) {
            const uint32_t pos = off + pre + __popc(bal & lt);
            kout[pos] = key;
            vout[pos] = (uint32_t)item;
        }
        off += cnt;
    }
    if (blockIdx.x == gridDim.x - 1) {
        uint32_t lo = 0xFFFFFFFFu, hi = 0u;
        for (int b = threadIdx.x; b < nblocks; b += 256) {
            const uint2 r = block_range[b];
            lo = umin(lo, r.x);
            hi = umax(hi, r.y);
        }
        lo = __reduce_min_sync(0xFFFFFFFFu, lo);
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);
        __shared__ uint2 wrange[8];
        if (lane == 0) wrange[w] = make_uint2(lo, hi);
        __syncthreads();
        if (threadIdx.x == 0) {
            uint2 r = wrange[0];
            for (int k = 1; k < 8; ++k) r = make_uint2(umin(r.x, wrange[k].x), umax(r.y, wrange[k].y));
            counts[0] = counts[1] = 0u;
            counts[8] = off;
            counts[11] = r.x;
            counts[12] = r.y;
        }
    }
}

// a b + c d with one rounding of nearly the exact sum: the two rounded products' errors come from
// fused multiply-adds (Kahan's difference of products; its error is at most 1.5 ulp of the result:
// Jeannerod, Louvet and Muller, Math. Comp. 82, 2013).
__device__ __forceinline__ float dot2(float a, float b, float c, float d) {
    const float p = __fmul_rn(c, d);
    return __fadd_rn(__fmaf_rn(a, b, p), __fmaf_rn(c, d, -p));
}

// Adjoint of the projection, one thread a Gaussian, all its views. The conic
// Q = (P S^2 P^T + dilation I)^-1, P = J W R the projected unit axes and S the scales, is taken back in
// the Gaussian's own axes: with x_k = Q p_k, X = (x_0 x_1 x_2) and the symmetric matrix Gc of the
// conic's gradient (g_a, g_c and half of g_b off the diagonal),
//   K_jk = -2 x_j^T Gc x_k          (twice dL/dSigma in body axes),
//   dL/dlog s_k = K_kk s_k^2,       torque about axis 0 = K_12 (s_1^2 - s_2^2), the others cyclically,
//   dL/dJ = -2 Q Gc X S^2 (W R)^T.
// For an elongated projection the determinant A C - B B of its covariance, the adjoint -Q Gc Q in
// terms of A, B, C, and the products with Sigma after it cancel almost fully in float32: errors of
// 1e-7 grew with the ratio of the axes' variances, and one such Gaussian near the camera could carry
// most of the error of the whole gradient. Here the determinant and the x_k come from the minors n of
// P as sums that do not cancel so:
//   det = d (d + A0 + C0) + s_1^2 s_2^2 n_0^2 + s_0^2 s_2^2 n_1^2 + s_0^2 s_1^2 n_2^2   (d the dilation),
//   det X = d P + (Q1 x n, -Q0 x n), Q0 and Q1 the rows of P S^2,
// and the two contractions that cancel by their nature (Gc x_k, x_j . Gc x_k) are dot2's. Error over
// the gradient's norm of 110 random room scenes in the deterministic mode: median 1.35e-6 -> 0.94e-6
// (what the forward's float32 covariance leaves), 2.8e-5 -> 6e-7 in the worst conditioned one, never
// above what it was; of thin Gaussians near the camera 1e-3 -> below 4e-5.
//
// Bound by its chain of dependent instructions: an item's gradients are loaded before the shape is
// formed, the statistics are added in L2 instead of read, and four CTAs an SM leave it the registers
// it wants (300k-Gaussian keyframe 22.7 -> 20.7 us, 8-view window of 150k 39.7 -> 37.3; five CTAs 20.7
// and 42.0, six 23.1 and 47.5 with their spills).
__global__ void __launch_bounds__(128, 4) k_preprocess_backward(
    const float* __restrict__ P, int n, int cap, int n_views, const DevCamera* __restrict__ cams, DevConst kc,
    const float* __restrict__ grad2d, const uint32_t* __restrict__ tiles, float* __restrict__ G,
    float* __restrict__ dens_sum, float* __restrict__ dens_cnt, const uint32_t* __restrict__ overflow, int add_reg,
    float reg_scale) {
    int gid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= n) return;
    float p[kParamRows];
    load_params(P, cap, gid, p);
    float dmu[3] = {0.f, 0.f, 0.f};
    float K[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // K_00, K_11, K_22, K_12, K_02, K_01
    float dop = 0.f, dr = 0.f, dg = 0.f, db = 0.f;
    float gsum = 0.f, gcnt = 0.f;
    // the screen gradients of the view at hand, where the Gaussian has tiles in it
    float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0;
    float g8 = 0.f;
    bool seen = false;
    auto load_view = [&](int view) {
        const size_t item = (size_t)view * n + gid;
        seen = tiles[item] != 0;
        if (seen) {
            g0 = *reinterpret_cast<const float4*>(grad2d + item * kGrad2dStride);
            g1 = *reinterpret_cast<const float4*>(grad2d + item * kGrad2dStride + 4);
            g8 = grad2d[item * kGrad2dStride + 8];
        }
    };
    load_view(0);
    float s[3], sq[3], R[9];
    {
        float q[4];
        rotation_of(p, q, R);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        s[k] = expf(p[3 + k]);
        sq[k] = s[k] * s[k];
    }
    for (int view = 0; view < n_views; ++view) {
        if (view > 0) load_view(view);
        if (!seen) continue;
        const DevCamera& cam = cams[view];
        // the compositing adjoint leaves out the factor ln 2 of the first five values; with the
        // exp2 scaling of the conic (a' = -a log2(e) / 2, b' = -b log2(e)) it cancels there
        float gu = g0.x * kLn2, gv = g0.y * kLn2;
        float ga = -0.5f * g0.z, gb = -g0.w, gc = -0.5f * g1.x;   // to the unscaled conic
        dop += g1.y;
        dr += g1.z;
        dg += g1.w;
        db += g8;
        {   // densification statistic: position-gradient norm in NDC (du/dx_ndc = W/2)
            const float nu = gu * (0.5f * (float)cam.width), nv = gv * (0.5f * (float)cam.height);
            gsum += sqrtf(nu * nu + nv * nv);
        }
        gcnt += 1.f;
        const float d = kc.dilation;
        const float tx = cam.R[0] * p[0] + cam.R[1] * p[1] + cam.R[2] * p[2] + cam.t[0];
        const float ty = cam.R[3] * p[0] + cam.R[4] * p[1] + cam.R[5] * p[2] + cam.t[1];
        const float tz = cam.R[6] * p[0] + cam.R[7] * p[1] + cam.R[8] * p[2] + cam.t[2];
        const float iz = 1.0f / tz, iz2 = iz * iz, iz3 = iz2 * iz;
        const float xr = tx * iz, yr = ty * iz;
        const float xh = fminf(fmaxf(xr, -cam.lim_x), cam.lim_x), yh = fminf(fmaxf(yr, -cam.lim_y), cam.lim_y);
        const float J00 = cam.fx * iz, J02 = -cam.fx * xh * iz, J11 = cam.fy * iz, J12 = -cam.fy * yh * iz;
        float Vm[3][3], p0[3], p1[3], q0[3], q1[3];   // V = W R, P = J V, P S^2
#pragma unroll
        for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
                Vm[r][k] = cam.R[3 * r] * R[k] + cam.R[3 * r + 1] * R[3 + k] + cam.R[3 * r + 2] * R[6 + k];
            p0[k] = J00 * Vm[0][k] + J02 * Vm[2][k];
            p1[k] = J11 * Vm[1][k] + J12 * Vm[2][k];
            q0[k] = sq[k] * p0[k];
            q1[k] = sq[k] * p1[k];
        }
        const float n0 = p0[1] * p1[2] - p0[2] * p1[1], n1 = p0[2] * p1[0] - p0[0] * p1[2],
                    n2 = p0[0] * p1[1] - p0[1] * p1[0];
        const float A0 = q0[0] * p0[0] + q0[1] * p0[1] + q0[2] * p0[2];   // A and C without the dilation
        const float C0 = q1[0] * p1[0] + q1[1] * p1[1] + q1[2] * p1[2];
        const float B = q0[0] * p1[0] + q0[1] * p1[1] + q0[2] * p1[2];
        const float det = d * (d + A0 + C0) + sq[1] * sq[2] * n0 * n0 + sq[0] * sq[2] * n1 * n1 +
                          sq[0] * sq[1] * n2 * n2;
        const float idet = 1.0f / fmaxf(det, 1e-37f);   // (zero only where everything it scales is)
        const float x0[3] = {(d * p0[0] + (q1[1] * n2 - q1[2] * n1)) * idet,
                             (d * p0[1] + (q1[2] * n0 - q1[0] * n2)) * idet,
                             (d * p0[2] + (q1[0] * n1 - q1[1] * n0)) * idet};
        const float x1[3] = {(d * p1[0] - (q0[1] * n2 - q0[2] * n1)) * idet,
                             (d * p1[1] - (q0[2] * n0 - q0[0] * n2)) * idet,
                             (d * p1[2] - (q0[0] * n1 - q0[1] * n0)) * idet};
        const float h = 0.5f * gb;
        float z0[3], z1[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            z0[k] = -2.f * dot2(ga, x0[k], h, x1[k]);
            z1[k] = -2.f * dot2(h, x0[k], gc, x1[k]);
        }
        K[0] += dot2(x0[0], z0[0], x1[0], z1[0]);
        K[1] += dot2(x0[1], z0[1], x1[1], z1[1]);
        K[2] += dot2(x0[2], z0[2], x1[2], z1[2]);
        K[3] += dot2(x0[1], z0[2], x1[1], z1[2]);
        K[4] += dot2(x0[0], z0[2], x1[0], z1[2]);
        K[5] += dot2(x0[0], z0[1], x1[0], z1[1]);
        // -2 Gc X S^2 (W R)^T, column by column of the camera's axes
        float e0[3], e1[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float f0 = Vm[r][0] * (sq[0] * x0[0]) + Vm[r][1] * (sq[1] * x0[1]) + Vm[r][2] * (sq[2] * x0[2]);
            const float f1 = Vm[r][0] * (sq[0] * x1[0]) + Vm[r][1] * (sq[1] * x1[1]) + Vm[r][2] * (sq[2] * x1[2]);
            e0[r] = -2.f * (ga * f0 + h * f1);
            e1[r] = -2.f * (h * f0 + gc * f1);
        }
        const float A = A0 + d, C = C0 + d;
        const float dJ00 = (C * e0[0] - B * e1[0]) * idet, dJ02 = (C * e0[2] - B * e1[2]) * idet;
        const float dJ11 = (A * e1[1] - B * e0[1]) * idet, dJ12 = (A * e1[2] - B * e0[2]) * idet;
        float dtx = 0.f, dty = 0.f, dtz = 0.f;
        dtz += -cam.fx * iz2 * dJ00 - cam.fy * iz2 * dJ11;
        if (fabsf(xr) <= cam.lim_x) {
            dtx += -cam.fx * iz2 * dJ02;
            dtz += 2.f * cam.fx * tx * iz3 * dJ02;
        } else {
            dtz += cam.fx * xh * iz2 * dJ02;
        }
        if (fabsf(yr) <= cam.lim_y) {
            dty += -cam.fy * iz2 * dJ12;
            dtz += 2.f * cam.fy * ty * iz3 * dJ12;
        } else {
            dtz += cam.fy * yh * iz2 * dJ12;
        }
        // screen mean u = fx tx/tz + cx, v = fy ty/tz + cy
        dtx += gu * cam.fx * iz;
        dty += gv * cam.fy * iz;
        dtz += -(gu * cam.fx * tx + gv * cam.fy * ty) * iz2;
        // t = W mu + t_w
        dmu[0] += cam.R[0] * dtx + cam.R[3] * dty + cam.R[6] * dtz;
        dmu[1] += cam.R[1] * dtx + cam.R[4] * dty + cam.R[7] * dtz;
        dmu[2] += cam.R[2] * dtx + cam.R[5] * dty + cam.R[8] * dtz;
    }
    float dls[3] = {K[0] * sq[0], K[1] * sq[1], K[2] * sq[2]};
    if (add_reg) {
        // Eq. 10 planar term: mean_i max(floor, min_k s_ik); gradient on the (first) smallest axis
        int km = 0;
        float sm = s[0];
        if (s[1] < sm) { sm = s[1]; km = 1; }
        if (s[2] < sm) { sm = s[2]; km = 2; }
        if (sm > kc.reg_floor) dls[km] += reg_scale * sm;
    }
    // R exp([omega]x) is the quaternion q (1, omega / 2): dL/dq = 2 q (0, torque), tangent to the unit
    // sphere, over |q| for the quaternion before its normalisation
    float q[4];
    const float qnorm = rotation_of(p, q, R);
    const float w = q[0], x = q[1], y = q[2], z = q[3];
    const float tw0 = K[3] * ((s[1] - s[2]) * (s[1] + s[2])), tw1 = K[4] * ((s[2] - s[0]) * (s[2] + s[0])),
                tw2 = K[5] * ((s[0] - s[1]) * (s[0] + s[1]));
    const float iq2 = 2.0f / qnorm;
    float oa = 1.0f / (1.0f + expf(-p[10]));
    size_t c = (size_t)cap;
    G[0 * c + gid] = dmu[0];
    G[1 * c + gid] = dmu[1];
    G[2 * c + gid] = dmu[2];
    G[3 * c + gid] = dls[0];
    G[4 * c + gid] = dls[1];
    G[5 * c + gid] = dls[2];
    G[6 * c + gid] = -(x * tw0 + y * tw1 + z * tw2) * iq2;
    G[7 * c + gid] = (w * tw0 + y * tw2 - z * tw1) * iq2;
    G[8 * c + gid] = (w * tw1 + z * tw0 - x * tw2) * iq2;
    G[9 * c + gid] = (w * tw2 + x * tw1 - y * tw0) * iq2;
    G[10 * c + gid] = dop * (1.f - oa);   // the records hold o dL/do, do/dlogit = o (1 - o)
    G[11 * c + gid] = dr;
    G[12 * c + gid] = dg;
    G[13 * c + gid] = db;
    if (dens_sum != nullptr && gcnt > 0.f && *overflow == 0u) {   // (an overflow: nothing was composited)
        atomicAdd(dens_sum + gid, gsum);   // (one each: added in L2, nothing waits for it)
        atomicAdd(dens_cnt + gid, gcnt);
    }
}

}  // namespace

// Projection of every (view, Gaussian) item; above the size that one CTA sorts, then the visible items
// compacted in item order into dkey[1] / dval[1] (their number in dcount[8], their keys' range in
// dcount[11], dcount[12]).
cudaError_t launch_preprocess(gs_ctx* c, int n_views, const DevConst& k, cudaStream_t s) {
    if (c->n == 0) return cudaSuccess;
    dim3 grid((c->n + 255) / 256, n_views);
    const uint32_t nblocks = grid.x * grid.y;
    ++c->launches;
    k_preprocess<<<grid, 256, 0, s>>>(c->params, c->n, c->cap, c->dcam, k, c->tile, c->rec, c->tiles_touched,
                                       c->dkey[0], c->depth, c->vis_blocks, c->vis_range,
                                       k.lambda_reg / (float)c->n, c->reg_part);
    if (!depth_sort_small(c)) {
        ++c->launches;
        k_compact_visible<<<(nblocks + kCompactSub - 1) / kCompactSub, 256, 0, s>>>(
            c->dkey[0], c->n, (int)grid.x, (int)nblocks, c->vis_blocks, c->vis_range, c->dkey[1], c->dval[1], c->dcount);
    }
    return cudaGetLastError();
}

cudaError_t launch_preprocess_backward(gs_ctx* c, const DevConst& k, bool add_reg, cudaStream_t s) {
    if (c->n == 0) return cudaSuccess;
    float reg_scale = k.lambda_reg / (float)c->n;
    ++c->launches;
    k_preprocess_backward<<<(c->n + 127) / 128, 128, 0, s>>>(c->params, c->n, c->cap, c->n_views, c->dcam, k,
                                                              c->grad2d, c->tiles_touched, c->grads, c->dens_sum,
                                                              c->dens_cnt, c->dcount + 9, add_reg ? 1 : 0, reg_scale);
    return cudaGetLastError();
}

}  // namespace gs
