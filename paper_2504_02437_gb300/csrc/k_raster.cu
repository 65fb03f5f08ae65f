// Front-to-back alpha compositing (Eq. 3, Section 3.1) and its adjoint.
//
// A persistent grid walks the (view, tile) work list; each thread owns PPT
// pixels of one column of its tile, and each warp an 8 x (4 PPT) pixel block, so
// a Gaussian that misses a warp's block costs that warp one test. The tile's
// sorted pair list is walked in batches of records staged in shared memory
// (gathered by Gaussian id from the 48-byte raster records).
//
// Two things bound a launch: the SMs' issue slots where tiles are many and alike,
// and the longest tile's chain of dependent visits where they are few or unlike
// (a 16 x 2 tile of a 1200x680 keyframe took one CTA 541 us while the average CTA
// was busy for 264). Whole tiles of two pixels a thread are written for the first
// (branches around pixels that are not hit); long tiles go as halves of one pixel
// a thread, written for the second (visits two at a time and without branches).
//
// Membership is pixel-exact (|px - u| <= r and |py - v| <= r), so the image is
// the same for every tile size: tiles only bound which Gaussians a pixel tests.
#include <algorithm>
#include <type_traits>

#include "gs_internal.cuh"

namespace gs {
namespace {

// records staged in shared memory per batch: 512 for CTAs of 128 or 256
// threads (fewer barriers per tile: on the 300k-Gaussian keyframe 2 % faster
// than 256 for 256 threads, 3 % for 128; 128 records were 7 % slower), 256 for
// CTAs of 64 threads (there 512 records limit the SM to 6 CTAs by shared memory
// and the 8-view window slows by 30 %)
constexpr int batch_for(int threads) { return threads >= 128 ? 512 : 256; }

// A Gaussian that at most this many lanes of a warp blended gets its 9
// gradient values added by each of those lanes (two float4 atomics and one
// scalar) instead of a 12-shuffle warp sum and one 9-lane atomic: fewer issue
// slots for the warp; past about half a warp the same-address atomics cost more
// (on the 300k-Gaussian keyframe, 16 x 2 layout: 7 % faster than a threshold of
// one lane, 24 about 1 % faster than 16 and 12; every lane, 2 % slower)
constexpr int kLaneAtomicMax = 24;

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Two floats in one 64-bit register and the packed IEEE operations on them (each half rounds as the
// scalar operation does): in the adjoint a thread's pixels go in pairs, one instruction for both, and
// a pixel that a Gaussian misses takes part with alpha 0 instead of branching around.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ F2 pack2(float a) { return pack2(a, a); }
__device__ __forceinline__ void unpack2(F2 x, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// A colour or an upstream gradient that is not finite, or so large that a product of two overflows:
// times a weight of zero it would not vanish, so a batch (or warp) with one masks its operands.
__device__ __forceinline__ bool unsafe(float x) { return !(fabsf(x) <= 1e15f); }

// A raster record staged for one tile, relative to the local origin (ox, oy),
// the tile's corner rounded down to a multiple of 32 px:
//   s0 = {u, v, hx, hy}: local screen mean and the half-widths of the pixel
//        box a pixel must lie in to be blended;
//   s1 = {a', b', c', o}: exp2-scaled conic and opacity;
//   s2 = {R, G, B, thr}: colour and the exponent threshold of the alpha cutoff.
// The screen mean is stored split (integer part in f0.xy, fractions in f1.w,
// f2.w); the local mean (ui - ox) + uf is formed once per pair and tile, so
// pixel offsets carry the rounding of a small number only, and the same for
// tiles of 8, 16 or 32 px (which keeps the image bit-identical across tile
// sizes).
//
// Blending needs |dx| <= r, |dy| <= r (the membership box) and
// o 2^p2 >= alpha_min, i.e. p2 >= thr = log2(alpha_min / o) with
// p2 = a' dx^2 + b' dx dy + c' dy^2 (negative definite). The set p2 >= thr is
// an ellipse whose axis-aligned half-widths are sqrt(-thr (B^-1)_xx),
// sqrt(-thr (B^-1)_yy) with B = -[[a', b'/2], [b'/2, c']]; hx, hy are those
// widths enlarged by 0.1 % + 0.01 px (far above float32 rounding) and capped
// at r, so a pixel outside (hx, hy) cannot blend and skipping it leaves the
// result unchanged. A Gaussian with o < alpha_min gets hx = hy = -1.
__device__ __forceinline__ void stage_record(const float4* __restrict__ rec, uint32_t item, float ox, float oy,
                                             float alpha_min, float4& s0, float4& s1, float4& s2) {
    const float4 a = rec[(size_t)item * 3 + 0];
    const float4 q = rec[(size_t)item * 3 + 1];
    const float4 c = rec[(size_t)item * 3 + 2];
    const float r = a.z, o = a.w;
    const float thr = log2f(alpha_min) - log2f(o);
    float hx = -1.f, hy = -1.f;
    if (thr <= 0.f) {
        const float det = q.x * q.z - 0.25f * q.y * q.y;
        if (det > 0.f) {
            const float kap = -thr / det;
            hx = fminf(fmaf(sqrtf(-kap * q.z), 1.001f, 0.01f), r);
            hy = fminf(fmaf(sqrtf(-kap * q.x), 1.001f, 0.01f), r);
        } else {
            hx = hy = r;
        }
    }
    s0 = make_float4((a.x - ox) + q.w, (a.y - oy) + c.w, hx, hy);
    s1 = make_float4(q.x, q.y, q.z, o);
    s2 = make_float4(c.x, c.y, c.z, thr);
}

// The same ellipse's extent across its long axis: with Q = -(a' dx^2 + b' dx dy + c' dy^2)
// = d^T M d, the set Q <= -thr has half-width sqrt(-thr / lambda_max(M)) along the unit
// eigenvector n of lambda_max(M) (the ellipse's short axis), enlarged by the same margin as the
// box. A pixel block whose projection on n lies farther from the mean cannot blend; for an
// elongated, rotated ellipse this strip cuts much of its axis-aligned box.
__device__ __forceinline__ void short_axis_strip(const float4 s1, float thr, float& nx, float& ny, float& wn) {
    nx = 1.f;
    ny = 0.f;
    wn = 3.0e38f;
    const float A = -s1.x, B2 = -0.5f * s1.y, C = -s1.z;   // M = [[A, B2], [B2, C]]
    if (!(thr <= 0.f)) return;
    const float half = 0.5f * (A - C);
    const float lam = 0.5f * (A + C) + sqrtf(half * half + B2 * B2);
    if (!(lam > 0.f)) return;
    // eigenvector of lam: the better conditioned of (B2, lam - A) and (lam - C, B2)
    float ex = B2, ey = lam - A;
    const float fx = lam - C, fy = B2;
    if (fx * fx + fy * fy > ex * ex + ey * ey) {
        ex = fx;
        ey = fy;
    }
    const float nn = ex * ex + ey * ey;
    if (!(nn > 0.f)) return;
    const float inv = rsqrtf(nn);
    nx = ex * inv;
    ny = ey * inv;
    wn = fmaf(sqrtf(-thr / lam), 1.001f, 0.01f);
}

// Thread layout of a work item, 1 / SPLIT of the rows of a TILE x TILE tile: each thread owns PPT
// pixels of one column, 4 rows apart; warp w owns an 8 x (4 PPT) block.
template <int TILE, int PPT, int SPLIT = 1>
struct Layout {
    static constexpr int kThreads = TILE * TILE / PPT / SPLIT;
    static constexpr int kRows = TILE / SPLIT;
    static constexpr int kBlocksX = TILE / 8;
    // resident CTAs per SM the fused kernel is compiled for (its register cap): 16 x 1 (8 warps a
    // CTA) capped at 64 registers for 4 CTAs instead of 3 (8-view 640x480 window: fused kernel
    // 0.748 -> 0.645 ms; 5 CTAs 0.652, 6 CTAs 0.716). 0 leaves the bound unset, so the others
    // keep the compiler's own register count (an explicit bound of 1 let it take more: 16 x 2
    // rose from 80 to 96 registers, 5 CTAs per SM instead of 6, 5 % slower)
    static constexpr int kMinBlocks = (TILE == 16 && PPT == 1) ? 4 : 0;
    // visit-list entries a thread of one pixel takes together: two in halves of long tiles, whose
    // latency counts (1200x680 keyframe with 300k Gaussians: fused kernel 362, 355 and 345 us for 1, 2
    // and 4; 8-view window 785 us with 2, 856 with 4), one where a launch is bound by issue slots
    // (16 x 1: 376, 398 and 427 us)
    static constexpr int kVisits = SPLIT == 2 ? 2 : 1;
    static constexpr int kVisitsDet = 4;   // (fused kernel 220, 204 and 197 us for 1, 2 and 4: three 321x243 views)
    // long tiles go as two items of one pixel a thread, in the same CTAs as whole tiles of two
    static constexpr bool kHalves = TILE == 16 && PPT == 2;
    // the adjoint reuses the forward's staged batch and visit lists when the tile's whole list
    // fits one batch, and then starts without CTA barriers (each warp cuts its own list at its
    // own end): 16 x 1 window 0.645 -> 0.634 ms, 8 x 1 0.653 -> 0.636 ms; not for 16 x 2, where
    // the warps' imbalance moves to the work queue's barrier (300k-Gaussian keyframe: 0.362 ->
    // 0.383 ms)
    static constexpr bool kReuseStaged = !(TILE == 16 && PPT == 2) && SPLIT == 1;
    __device__ static void pixel(int tid, int& lx, int& ly0) {
        const int w = tid >> 5, l = tid & 31;
        lx = (w % kBlocksX) * 8 + (l & 7);
        ly0 = (w / kBlocksX) * (4 * PPT) + (l >> 3);
    }
};

// Base-2 exponent a' dx^2 + b' dx dy + c' dy^2 of a Gaussian at a pixel, as a
// polynomial in dy: (c' dy + b' dx) dy + a' dx^2, with the column terms
// b' dx and a' dx^2 formed once per (thread, Gaussian) and shared by the
// thread's pixels; two fused multiply-adds per pixel. Written with explicit
// rounding so that every kernel takes bit-identical decisions.
__device__ __forceinline__ float power2_dy(float qz, float qydx, float qxdx2, float dy) {
    return __fmaf_rn(__fmaf_rn(qz, dy, qydx), dy, qxdx2);
}

// Warp sum of 9 values by recursive halving: at each step a lane keeps half of
// its values and trades the other half with its partner, so 9 values cost 11
// exchanges instead of 45. Afterwards even lane L holds the full sum of value
// *idx (or idx = -1 if its slot is padding); each value sits in exactly one
// even lane.
__device__ __forceinline__ float warp_sum9(const float (&v)[9], int lane, int& idx) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    float w[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const float a = v[i], b = (i + 5 < 9) ? v[i + 5] : 0.f;
        w[i] = (b4 ? b : a) + __shfl_xor_sync(0xFFFFFFFFu, b4 ? a : b, 16);
    }
    float x[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float a = w[i], b = (i + 3 < 5) ? w[i + 3] : 0.f;
        x[i] = (b3 ? b : a) + __shfl_xor_sync(0xFFFFFFFFu, b3 ? a : b, 8);
    }
    float y[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float a = x[i], b = (i + 2 < 3) ? x[i + 2] : 0.f;
        y[i] = (b2 ? b : a) + __shfl_xor_sync(0xFFFFFFFFu, b2 ? a : b, 4);
    }
    float z = (b1 ? y[1] : y[0]) + __shfl_xor_sync(0xFFFFFFFFu, b1 ? y[0] : y[1], 2);
    z += __shfl_xor_sync(0xFFFFFFFFu, z, 1);
    const int s3 = b2 ? 2 : 0, s4 = b1 ? 1 : 0;
    const int local = (b3 ? 3 : 0) + s3 + s4;
    const int id = (b4 ? 5 : 0) + local;
    idx = ((lane & 1) == 0 && s3 + s4 < 3 && local < 5 && id < 9) ? id : -1;
    return z;
}

// Shared-memory staging of one batch of B raster records for a CTA of NW
// warps, shared by the forward and backward passes.
template <int B, int NW>
struct Stage {
    // index of an entry of a staged batch
    typedef typename std::conditional<B <= 256, uint8_t, uint16_t>::type Idx;
    float4 s0[B], s1[B], s2[B];
    uint32_t sid[B];
    uint32_t mask[B];   // bit w: the record's pixel box meets warp w's pixel block
    Idx list[NW][B];   // per warp: the batch entries it must visit, in order
};

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Compacts the entries k < cnt of the staged batch whose mask has this warp's
// bit (and, when `limit` is given, lie before it) into the warp's list, in
// ascending order; returns their number. Called by all 32 lanes of the warp.
template <int B, int NW>
__device__ __forceinline__ int build_warp_list(Stage<B, NW>& st, int cnt, uint32_t base, uint32_t limit) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t wbit = 1u << w, lt = lanemask_lt();
    int nk = 0;
    for (int c0 = 0; c0 < cnt; c0 += 32) {
        const int k = c0 + lane;
        const bool hit = k < cnt && (st.mask[k] & wbit) && base + (uint32_t)k < limit;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, hit);
        if (hit) st.list[w][nk + __popc(bal & lt)] = (typename Stage<B, NW>::Idx)k;
        nk += __popc(bal);
    }
    __syncwarp();
    return nk;
}
template <int B, int NW>
__device__ __forceinline__ Stage<B, NW>& stage() {
    __shared__ Stage<B, NW> st;
    return st;
}

// Geometry of one work item (a tile of one view) as seen by one thread.
template <int TILE, int PPT, int SPLIT = 1>
struct TileGeom {
    int view, txi, row0, px, py0;
    float ox, oy, fx;
    uint2 rg;
    __device__ TileGeom(int bin, int part, const uint2* __restrict__ ranges, int tiles_x, int tiles_per_view) {
        view = bin / tiles_per_view;
        const int t = bin - view * tiles_per_view;
        const int tyi = t / tiles_x;
        txi = t - tyi * tiles_x;
        int lx, ly0;
        Layout<TILE, PPT, SPLIT>::pixel(threadIdx.x, lx, ly0);
        px = txi * TILE + lx;
        row0 = tyi * TILE + part * Layout<TILE, PPT, SPLIT>::kRows;
        py0 = row0 + ly0;
        // pixel offsets are taken from a 32-px-aligned local origin (see load_record)
        ox = (float)((txi * TILE) & ~31);
        oy = (float)((tyi * TILE) & ~31);
        fx = (float)px - ox;
        rg = ranges[bin];
    }
    __device__ int py(int p) const { return py0 + 4 * p; }
};

// Warps of the CTA whose 8 x (4 PPT) pixel block meets the box u +- hx, v +- hy and the
// short-axis strip |n . (x - u)| <= wn.
template <int TILE, int PPT, int SPLIT>
__device__ __forceinline__ uint32_t warp_mask(const TileGeom<TILE, PPT, SPLIT>& g, const float4 s0, const float4 s1,
                                              float thr) {
    float nx, ny, wn;
    short_axis_strip(s1, thr, nx, ny, wn);
    // half-extents of a warp's pixel block projected on n, plus the rounding slack of the box test
    const float hb = 3.5f * fabsf(nx) + 0.5f * (float)(4 * PPT - 1) * fabsf(ny) + wn + 0.01f;
    constexpr int NW = Layout<TILE, PPT, SPLIT>::kThreads / 32;
    constexpr int BX = Layout<TILE, PPT, SPLIT>::kBlocksX;
    const float tox = (float)(g.txi * TILE) - g.ox, toy = (float)g.row0 - g.oy;
    // widened by 0.01 px so that rounding cannot drop a pixel the per-pixel test would keep
    const float x0 = s0.x - s0.z - 0.01f, x1 = s0.x + s0.z + 0.01f, y0 = s0.y - s0.w - 0.01f,
                y1 = s0.y + s0.w + 0.01f;
    uint32_t m = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const float bx = tox + 8.f * (float)(w % BX), by = toy + (float)(4 * PPT) * (float)(w / BX);
        const float sc = nx * (bx + 3.5f - s0.x) + ny * (by + 0.5f * (float)(4 * PPT - 1) - s0.y);
        const bool hit = x0 <= bx + 7.f && x1 >= bx && y0 <= by + (float)(4 * PPT - 1) && y1 >= by && fabsf(sc) <= hb;
        m |= hit ? (1u << w) : 0u;
    }
    return m;
}

// Forward compositing (Eq. 3) of a thread's PPT pixels over the tile's sorted
// list. Returns final T, the colour, and per pixel the number of list entries
// up to and including the last blended Gaussian; optionally the Eq. 8 argmax.
// The return value is the length of the warp's visit list when the tile's whole
// list was staged as one batch (it is left in shared memory for the adjoint),
// else -1; which of the two is the same for every warp of the CTA.
template <int TILE, int PPT, int SPLIT, bool ARGMAX, bool DET>
__device__ __forceinline__ int fwd_core(const TileGeom<TILE, PPT, SPLIT>& g, const bool (&inside)[PPT],
                                         const uint32_t* __restrict__ pval, const uint32_t* __restrict__ emit_item,
                                         const float4* __restrict__ rec, const DevConst& kc, float (&T)[PPT], float (&cr)[PPT], float (&cg)[PPT],
                                         float (&cb)[PPT], uint32_t (&last)[PPT], uint32_t (&amax)[PPT],
                                         bool& masked) {
    constexpr int NT = Layout<TILE, PPT, SPLIT>::kThreads;
    constexpr int kBatch = batch_for(NT);
    Stage<kBatch, NT / 32>& st = stage<kBatch, NT / 32>();
    float4* s0 = st.s0;
    float4* s1 = st.s1;
    float4* s2 = st.s2;
    uint32_t* sid = st.sid;
    // a pixel that is outside the image or has stopped gets a row offset so far away that it
    // fails every box test (and its exponent is -inf): no separate per-pixel flag to test
    constexpr float kGone = 3.0e38f;
    float fy[PPT], wmax[PPT];
    int nlive = 0;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        fy[p] = inside[p] ? (float)g.py(p) - g.oy : kGone;
        nlive += inside[p] ? 1 : 0;
        T[p] = 1.f;
        cr[p] = cg[p] = cb[p] = 0.f;
        last[p] = 0;
        wmax[p] = -1.f;
        amax[p] = 0xFFFFFFFFu;
    }
    const uint2 rg = g.rg;
    int staged = -1;
    // for an adjoint that reuses the staged batch: whether its colours need masking there
    constexpr bool kMarkWild = !DET && Layout<TILE, PPT, SPLIT>::kReuseStaged;
    masked = false;
    for (uint32_t bs = rg.x; bs < rg.y; bs += kBatch) {
        if (__syncthreads_count(nlive > 0) == 0) break;
        bool wild = false;
        for (int i = threadIdx.x; i < kBatch; i += NT) {
            const uint32_t j = bs + i;
            if (j < rg.y) {
                const uint32_t pv = pval[j];   // the item, or its emission index (deterministic mode)
                const uint32_t item = DET ? emit_item[pv] : pv;
                stage_record(rec, item, g.ox, g.oy, kc.alpha_min, s0[i], s1[i], s2[i]);
                sid[i] = pv;
                st.mask[i] = warp_mask(g, s0[i], s1[i], s2[i].w);
                if constexpr (kMarkWild) wild |= unsafe(s2[i].x) || unsafe(s2[i].y) || unsafe(s2[i].z);
            }
        }
        if constexpr (kMarkWild)
            masked = __syncthreads_or(wild);
        else
            __syncthreads();
        const int cnt = min((uint32_t)kBatch, rg.y - bs);
        const int nk = build_warp_list(st, cnt, 0u, 0xFFFFFFFFu);
        if (rg.y - rg.x <= (uint32_t)kBatch) staged = nk;
        const typename Stage<kBatch, NT / 32>::Idx* wl = st.list[threadIdx.x >> 5];
        if constexpr (PPT == 1 || DET) {
            // U entries at a time, their loads, tests and alphas without branches, so that their
            // latencies overlap; only T runs through them in turn (16 x 1, one entry at a time, with
            // the adjoint in the same form: 1200x680 keyframe 416 -> 376 us, 160x120 47 -> 36 us; in
            // the deterministic mode, whose one warp a tile takes as long as its list, four at a time)
            constexpr int U = DET ? Layout<TILE, PPT, SPLIT>::kVisitsDet : Layout<TILE, PPT, SPLIT>::kVisits;
            bool live[PPT];
#pragma unroll
            for (int p = 0; p < PPT; ++p) live[p] = fy[p] != kGone;
            for (int i = 0; i < nk; i += U) {
                if (!__any_sync(0xFFFFFFFFu, nlive > 0)) break;
                int k[U];
                float al[U][PPT];
                bool hit[U][PPT];
                float4 c[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    k[u] = (int)wl[i + u] & (kBatch - 1);   // past nk: any entry, not hit
                    const float4 a = s0[k[u]], q = s1[k[u]];
                    c[u] = s2[k[u]];
                    const float dx = g.fx - a.x;
                    const float qydx = __fmul_rn(q.y, dx), qxdx2 = __fmul_rn(__fmul_rn(q.x, dx), dx);
                    const bool col = i + u < nk && fabsf(dx) <= a.z;
#pragma unroll
                    for (int p = 0; p < PPT; ++p) {
                        const float dy = fy[p] - a.y;
                        const float p2 = power2_dy(q.z, qydx, qxdx2, dy);
                        hit[u][p] = col && fabsf(dy) <= a.w && p2 >= c[u].w;
                        al[u][p] = fminf(kc.alpha_max, __fmul_rn(q.w, ex2_approx(p2)));
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
#pragma unroll
                    for (int p = 0; p < PPT; ++p) {
                        const float Tn = __fmul_rn(T[p], 1.f - al[u][p]);
                        const bool in = hit[u][p] && live[p];
                        const bool stop = in && Tn < kc.T_min;   // a pixel stops before it falls below T_min
                        live[p] = live[p] && !stop;
                        nlive -= stop ? 1 : 0;
                        if (in && live[p]) {
                            const float wgt = al[u][p] * T[p];
                            cr[p] = fmaf(c[u].x, wgt, cr[p]);
                            cg[p] = fmaf(c[u].y, wgt, cg[p]);
                            cb[p] = fmaf(c[u].z, wgt, cb[p]);
                            T[p] = Tn;
                            last[p] = bs + k[u] - rg.x + 1;
                            if (ARGMAX && wgt > wmax[p]) {
                                wmax[p] = wgt;
                                amax[p] = DET ? emit_item[sid[k[u]]] : sid[k[u]];
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < PPT; ++p) fy[p] = live[p] ? fy[p] : kGone;
            continue;
        }
        int knext = nk > 0 ? (int)wl[0] : 0;   // the next entry's index is loaded one visit ahead
        // unrolled by two: the next entry's record loads and membership tests interleave with
        // this entry's blending (A/B on the 300k-Gaussian keyframe, 16 x 2 layout: fused kernel
        // 0.380 -> 0.362 ms; the other layouts and the window unchanged; by four no better)
#pragma unroll 2
        for (int i = 0; i < nk && nlive > 0; ++i) {
            const int k = knext;
            if (i + 1 < nk) knext = wl[i + 1];
            const float4 a = s0[k];
            const float dx = g.fx - a.x;
            if (fabsf(dx) > a.z) continue;
            const float4 q = s1[k];
            const float thr = s2[k].w;
            const float qydx = __fmul_rn(q.y, dx), qxdx2 = __fmul_rn(__fmul_rn(q.x, dx), dx);
            // exponent and membership of every pixel first, without branches, so the
            // pixels' dependent chains interleave (5 % on the 300k-Gaussian keyframe
            // together with the same split in the adjoint)
            float p2v[PPT];
            bool hit[PPT];
            bool any_hit = false;
#pragma unroll
            for (int p = 0; p < PPT; ++p) {
                const float dy = fy[p] - a.y;
                p2v[p] = power2_dy(q.z, qydx, qxdx2, dy);
                hit[p] = fabsf(dy) <= a.w && p2v[p] >= thr;
                any_hit |= hit[p];
            }
            if (!any_hit) continue;
#pragma unroll
            for (int p = 0; p < PPT; ++p) {
                if (!hit[p]) continue;
                const float alpha = fminf(kc.alpha_max, __fmul_rn(q.w, ex2_approx(p2v[p])));
                const float Tn = __fmul_rn(T[p], 1.f - alpha);
                if (Tn < kc.T_min) {
                    fy[p] = kGone;
                    --nlive;
                    continue;
                }
                const float wgt = alpha * T[p];
                const float4 c = s2[k];
                cr[p] = fmaf(c.x, wgt, cr[p]);
                cg[p] = fmaf(c.y, wgt, cg[p]);
                cb[p] = fmaf(c.z, wgt, cb[p]);
                T[p] = Tn;
                last[p] = bs + k - rg.x + 1;
                if (ARGMAX && wgt > wmax[p]) {
                    wmax[p] = wgt;
                    amax[p] = DET ? emit_item[sid[k]] : sid[k];
                }
            }
        }
    }
    return staged;
}

// The nine screen partials of one Gaussian from a thread's sums of g2 = dL/dp2 (without ln 2),
// g2 dy, g2 dy^2 and minus the colour gradients over pixels that share dx: u, v, a', b', c', the
// opacity's times the opacity (its readers divide), r, g, b.
__device__ __forceinline__ void screen_partials(const float4 q, float dx, float g2, float g2y, float g2yy, float ncr,
                                                float ncg, float ncb, float (&acc)[9]) {
    acc[0] = -fmaf(2.f * q.x * dx, g2, q.y * g2y);
    acc[1] = -fmaf(q.y * dx, g2, 2.f * q.z * g2y);
    acc[2] = dx * dx * g2;
    acc[3] = dx * g2y;
    acc[4] = g2yy;
    acc[5] = g2;
    acc[6] = -ncr;
    acc[7] = -ncg;
    acc[8] = -ncb;
}

// Adds a warp's partials of one Gaussian (lanes with `any` blended it) to its record.
template <bool DET>
__device__ __forceinline__ void add_gradient(bool any, const float (&acc)[9], uint32_t id, int lane,
                                             float* __restrict__ grad2d, float* __restrict__ pairgrad) {
    const uint32_t who = __ballot_sync(0xFFFFFFFFu, any);
    if (who == 0u) return;
    if constexpr (DET) {
        // deterministic mode (one warp per tile): the warp's fixed-order sum is the
        // whole tile's contribution; it goes to the pair's own slot, no atomics
        int idx;
        const float v = warp_sum9(acc, lane, idx);
        if (idx >= 0) pairgrad[(size_t)id * kPairGradStride + idx] = v;
    } else if (__popc(who) <= kLaneAtomicMax) {
        // few lanes blended this Gaussian: each adds its own values (no warp sum)
        if (any) {
            float* gp = grad2d + (size_t)id * kGrad2dStride;
            atomicAdd(reinterpret_cast<float4*>(gp), make_float4(acc[0], acc[1], acc[2], acc[3]));
            atomicAdd(reinterpret_cast<float4*>(gp + 4), make_float4(acc[4], acc[5], acc[6], acc[7]));
            atomicAdd(gp + 8, acc[8]);
        }
    } else {
        int idx;
        const float v = warp_sum9(acc, lane, idx);
        if (idx >= 0) atomicAdd(grad2d + (size_t)id * kGrad2dStride + idx, v);
    }
}

// Adjoint of the compositing for a thread's PPT pixels: walks the tile's list
// back to front from the block's largest last-blended entry, recovering
// T_i = T_{i+1} / (1 - alpha_i) from the final T, and accumulates the
// gradients w.r.t. each Gaussian's screen quantities (the first five, u, v and
// the exp2-scaled conic a', b', c', without the factor ln 2 of d 2^p / dp; the opacity's times
// the opacity) (when at most
// kLaneAtomicMax lanes blended it, each adds its own 9 values with two float4
// atomics and one scalar; else a warp sum, then one 9-lane atomic). Each
// warp visits only the batch entries its compacted list holds, which stop at
// the warp's largest last-blended entry. With staged >= 0 (the forward left the
// tile's whole list staged, and this warp's visit list of that length) each
// warp cuts its own list at its own end and walks it without a CTA barrier.
template <int TILE, int PPT, int SPLIT, bool DET>
__device__ __forceinline__ void bwd_core(const TileGeom<TILE, PPT, SPLIT>& g, const uint32_t* __restrict__ pval,
                                         const uint32_t* __restrict__ emit_item, const float4* __restrict__ rec,
                                         const DevConst& kc, float (&T)[PPT], const uint32_t (&cnt_last)[PPT],
                                         const float (&gr)[PPT], const float (&gg)[PPT], const float (&gb)[PPT],
                                         float* __restrict__ grad2d, float* __restrict__ pairgrad, int staged,
                                         bool fwd_masks, bool masked) {
    constexpr int NT = Layout<TILE, PPT, SPLIT>::kThreads;
    constexpr int kBatch = batch_for(NT);
    Stage<kBatch, NT / 32>& st = stage<kBatch, NT / 32>();
    float4* s0 = st.s0;
    float4* s1 = st.s1;
    float4* s2 = st.s2;
    uint32_t* sid = st.sid;
    __shared__ uint32_t smax;
    const int lane = threadIdx.x & 31;
    const uint2 rg = g.rg;
    float fy[PPT], ga[PPT];   // ga: minus the upstream gradient . normalised colour behind the Gaussian
    uint32_t my_end[PPT];
    uint32_t thread_end = rg.x;
    bool wild = false;
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        fy[p] = (float)g.py(p) - g.oy;
        ga[p] = 0.f;
        wild |= unsafe(gr[p]) || unsafe(gg[p]) || unsafe(gb[p]);
        my_end[p] = rg.x + cnt_last[p];
        thread_end = max(thread_end, my_end[p]);
    }
    const uint32_t wm = __reduce_max_sync(0xFFFFFFFFu, thread_end);
    uint32_t end = wm;
    if (staged < 0) {   // the CTA's largest end decides which batches are staged again
        __syncthreads();
        if (threadIdx.x == 0) smax = rg.x;
        __syncthreads();
        if (lane == 0) atomicMax(&smax, wm);
        __syncthreads();
        end = smax;
    }
    const uint32_t warp_end = wm;
    const bool warp_wild = __any_sync(0xFFFFFFFFu, wild);
    for (uint32_t be = end; be > rg.x;) {
        const uint32_t bs = be - rg.x > (uint32_t)kBatch ? be - kBatch : rg.x;
        const typename Stage<kBatch, NT / 32>::Idx* wl = st.list[threadIdx.x >> 5];
        int nk;
        if (staged >= 0) {
            // the forward's visit list (ascending) is still staged: cut it before the warp's end
            int lo = 0, hi = staged;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (bs + (uint32_t)wl[mid] < warp_end) lo = mid + 1;
                else hi = mid;
            }
            nk = lo;
        } else {
            // the forward's warp masks of a one-batch tile are still staged (nothing writes them
            // in between): only the records are staged again
            const bool keep_masks = fwd_masks && rg.y - rg.x <= (uint32_t)kBatch;
            wild = false;
            __syncthreads();
            for (int i = threadIdx.x; i < kBatch; i += NT) {
                const uint32_t j = bs + i;
                if (j < be) {
                    const uint32_t pv = pval[j];   // the item, or its emission index (deterministic mode)
                    const uint32_t item = DET ? emit_item[pv] : pv;
                    stage_record(rec, item, g.ox, g.oy, kc.alpha_min, s0[i], s1[i], s2[i]);
                    sid[i] = pv;
                    if (!keep_masks) st.mask[i] = warp_mask(g, s0[i], s1[i], s2[i].w);
                    wild |= unsafe(s2[i].x) || unsafe(s2[i].y) || unsafe(s2[i].z);
                }
            }
            masked = __syncthreads_or(wild);
            nk = build_warp_list(st, (int)(be - bs), bs, warp_end);
        }
        if constexpr (PPT == 1 || DET) {
            // U entries at a time: their loads, tests and alphas first and without branches (a pixel that
            // is not hit has alpha 0 and adds zeros), then T and g . a through them in turn, then their sums
            constexpr int U = DET ? Layout<TILE, PPT, SPLIT>::kVisitsDet : Layout<TILE, PPT, SPLIT>::kVisits;
            for (int i = nk - 1; i >= 0; i -= U) {
                int k[U];
                bool any[U];
                float acc[U][9];
                float4 c[U], q[U];
                float dx[U], dy[U][PPT], oG[U][PPT], nal[U][PPT], rc[U][PPT];
                bool hit[U][PPT];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    k[u] = (int)wl[U == 1 ? i : max(i - u, 0)];
                    const float4 a = s0[k[u]];
                    q[u] = s1[k[u]];
                    c[u] = s2[k[u]];
                    dx[u] = g.fx - a.x;
                    const float qydx = __fmul_rn(q[u].y, dx[u]), qxdx2 = __fmul_rn(__fmul_rn(q[u].x, dx[u]), dx[u]);
                    const bool col = (U == 1 || i - u >= 0) && fabsf(dx[u]) <= a.z;
                    any[u] = false;
#pragma unroll
                    for (int p = 0; p < PPT; ++p) {
                        dy[u][p] = fy[p] - a.y;
                        const float p2 = power2_dy(q[u].z, qydx, qxdx2, dy[u][p]);
                        hit[u][p] = col && bs + k[u] < my_end[p] && fabsf(dy[u][p]) <= a.w && p2 >= c[u].w;
                        any[u] |= hit[u][p];
                        oG[u][p] = __fmul_rn(q[u].w, ex2_approx(p2));
                        nal[u][p] = hit[u][p] ? -fminf(kc.alpha_max, oG[u][p]) : 0.f;
                        rc[u][p] = rcp_approx(1.f + nal[u][p]);   // 1 - alpha >= 1 - alpha_max = 0.01
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float g2s = 0.f, g2y = 0.f, g2yy = 0.f, ncr = 0.f, ncg = 0.f, ncb = 0.f;
#pragma unroll
                    for (int p = 0; p < PPT; ++p) {
                        float gx = gr[p], gy = gg[p], gz = gb[p];
                        if ((masked | warp_wild) && !hit[u][p]) gx = gy = gz = 0.f;
                        T[p] *= rc[u][p];   // transmittance in front of this Gaussian
                        const float nw = nal[u][p] * T[p];
                        // dL/dalpha = T (g . c - g . a), with a the normalised colour behind this
                        // Gaussian, a <- a + alpha (c - a); g is fixed per pixel, so only -g . a is kept
                        const float d = fmaf(gx, c[u].x, fmaf(gy, c[u].y, gz * c[u].z)) + ga[p];
                        ga[p] = hit[u][p] ? fmaf(nal[u][p], d, ga[p]) : ga[p];
                        // through alpha = o 2^p2, zero where the 0.99 clamp holds; the factor ln 2
                        // of d(2^p2)/dp2 is left to the readers of the screen gradients
                        const float g2 = hit[u][p] && oG[u][p] <= kc.alpha_max ? T[p] * d * oG[u][p] : 0.f;
                        const float y = g2 * dy[u][p];
                        g2s += g2;
                        g2y += y;
                        g2yy = fmaf(y, dy[u][p], g2yy);
                        ncr = fmaf(nw, gx, ncr);
                        ncg = fmaf(nw, gy, ncg);
                        ncb = fmaf(nw, gz, ncb);
                    }
                    screen_partials(q[u], dx[u], g2s, g2y, g2yy, ncr, ncg, ncb, acc[u]);
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    add_gradient<DET>(any[u], acc[u], sid[k[u]], lane, grad2d, pairgrad);
            }
        } else {
            int knext = nk > 0 ? (int)wl[nk - 1] : 0;   // as in the forward: one visit ahead
            for (int i = nk - 1; i >= 0; --i) {
                const int k = knext;
                if (i > 0) knext = wl[i - 1];
                const uint32_t pos = bs + k;
                const float4 a = s0[k];
                const float dx = g.fx - a.x;
                // sums over the thread's pixels, which share dx: g2 = dL/dp2 (without ln 2), g2 dy,
                // g2 dy^2, and minus the colour gradients; the nine screen partials follow from them
                float g2s = 0.f, g2y = 0.f, g2yy = 0.f, ncr = 0.f, ncg = 0.f, ncb = 0.f;
                bool any = false;
                float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                if (fabsf(dx) <= a.z && pos < thread_end) {
                    q = s1[k];
                    const float4 c = s2[k];
                    const float qydx = __fmul_rn(q.y, dx), qxdx2 = __fmul_rn(__fmul_rn(q.x, dx), dx);
                    // the pixels in pairs; one that is not hit has alpha 0 and adds zeros (16 x 2 fused
                    // kernel against a branch per pixel: 1200x680 keyframe 348 -> 343 us, 8 x 640x480
                    // window of small splats 837 -> 792 us; the same in the forward was 4 % slower)
                    F2 dyv[PPT / 2];
                    float p2v[PPT];
                    bool hit[PPT];
#pragma unroll
                    for (int p = 0; p + 1 < PPT; p += 2) {
                        dyv[p / 2] = add2(pack2(fy[p], fy[p + 1]), pack2(-a.y));
                        const F2 pw = fma2(fma2(pack2(q.z), dyv[p / 2], pack2(qydx)), dyv[p / 2], pack2(qxdx2));
                        float dy0, dy1;
                        unpack2(dyv[p / 2], dy0, dy1);
                        unpack2(pw, p2v[p], p2v[p + 1]);
                        hit[p] = pos < my_end[p] && fabsf(dy0) <= a.w && p2v[p] >= c.w;
                        hit[p + 1] = pos < my_end[p + 1] && fabsf(dy1) <= a.w && p2v[p + 1] >= c.w;
                        any |= hit[p] | hit[p + 1];
                    }
                    if (any) {
#pragma unroll
                        for (int p = 0; p + 1 < PPT; p += 2) {
                            const F2 oG = mul2(pack2(q.w), pack2(ex2_approx(p2v[p]), ex2_approx(p2v[p + 1])));
                            float oG0, oG1;
                            unpack2(oG, oG0, oG1);
                            const F2 nal = pack2(hit[p] ? -fminf(kc.alpha_max, oG0) : 0.f,
                                                 hit[p + 1] ? -fminf(kc.alpha_max, oG1) : 0.f);
                            float om0, om1;
                            unpack2(add2(pack2(1.f), nal), om0, om1);
                            const F2 Tp = mul2(pack2(T[p], T[p + 1]), pack2(rcp_approx(om0), rcp_approx(om1)));
                            unpack2(Tp, T[p], T[p + 1]);
                            float g0r = gr[p], g1r = gr[p + 1], g0g = gg[p], g1g = gg[p + 1], g0b = gb[p],
                                  g1b = gb[p + 1];
                            F2 cx = pack2(c.x), cy = pack2(c.y), cz = pack2(c.z);
                            if (masked | warp_wild) {
                                cx = pack2(hit[p] ? c.x : 0.f, hit[p + 1] ? c.x : 0.f);
                                cy = pack2(hit[p] ? c.y : 0.f, hit[p + 1] ? c.y : 0.f);
                                cz = pack2(hit[p] ? c.z : 0.f, hit[p + 1] ? c.z : 0.f);
                                if (!hit[p]) g0r = g0g = g0b = 0.f;
                                if (!hit[p + 1]) g1r = g1g = g1b = 0.f;
                            }
                            const F2 nw = mul2(nal, Tp);
                            float nw0, nw1;
                            unpack2(nw, nw0, nw1);
                            ncr = fmaf(nw0, g0r, fmaf(nw1, g1r, ncr));
                            ncg = fmaf(nw0, g0g, fmaf(nw1, g1g, ncg));
                            ncb = fmaf(nw0, g0b, fmaf(nw1, g1b, ncb));
                            // dL/dalpha and g . a as for one pixel a thread
                            const F2 gap = pack2(ga[p], ga[p + 1]);
                            const F2 d = add2(fma2(pack2(g0r, g1r), cx, fma2(pack2(g0g, g1g), cy,
                                                                              mul2(pack2(g0b, g1b), cz))), gap);
                            unpack2(fma2(nal, d, gap), ga[p], ga[p + 1]);
                            float t0, t1;
                            unpack2(mul2(mul2(Tp, d), oG), t0, t1);
                            t0 = hit[p] && oG0 <= kc.alpha_max ? t0 : 0.f;
                            t1 = hit[p + 1] && oG1 <= kc.alpha_max ? t1 : 0.f;
                            float y0, y1, dy0, dy1;
                            unpack2(dyv[p / 2], dy0, dy1);
                            unpack2(mul2(pack2(t0, t1), dyv[p / 2]), y0, y1);
                            g2s += t0 + t1;
                            g2y += y0 + y1;
                            g2yy = fmaf(y0, dy0, fmaf(y1, dy1, g2yy));
                        }
                    }
                }
                float acc[9];
                screen_partials(q, dx, g2s, g2y, g2yy, ncr, ncg, ncb, acc);
                add_gradient<DET>(any, acc, sid[k], lane, grad2d, pairgrad);
            }
        }
        be = bs;
    }
}

// Persistent compositing kernels: a grid sized to the GPU's resident capacity
// walks the list of work items (tiles, or halves of tiles with long pair lists)
// through an atomic counter, so the load stays balanced across tiles of very
// different cost and across the views of a window. order[0] is the number of
// items, order[1 ..] the items: a bin, with the half plus one above kItemShift.
__device__ __forceinline__ bool next_work(uint32_t* __restrict__ queue, const uint32_t* __restrict__ order,
                                          int& bin, int& half) {
    __shared__ uint32_t s_work;
    __syncthreads();
    if (threadIdx.x == 0) {
        const uint32_t w = atomicAdd(queue, 1u);
        s_work = w < order[0] ? order[1 + w] : 0xFFFFFFFFu;
    }
    __syncthreads();
    const uint32_t w = s_work;
    if (w == 0xFFFFFFFFu) return false;
    bin = (int)(w & kItemBin);
    half = (int)(w >> kItemShift) - 1;
    return true;
}

template <int TILE, int PPT, int SPLIT>
__device__ __forceinline__ void inside_mask(const TileGeom<TILE, PPT, SPLIT>& g, int width, int height, bool (&inside)[PPT]) {
#pragma unroll
    for (int p = 0; p < PPT; ++p) inside[p] = g.px < width && g.py(p) < height;
}

// One work item's forward pass.
template <int TILE, int PPT, int SPLIT, bool ARGMAX, bool DET>
__device__ __forceinline__ void fwd_item(int bin, int part, const uint2* __restrict__ ranges,
                                         const uint32_t* __restrict__ pval, const float4* __restrict__ rec, int width,
                                         int height, int tiles_x, int tiles_per_view, int n, const DevConst& kc,
                                         float* __restrict__ out_rgb, float* __restrict__ out_T,
                                         uint32_t* __restrict__ out_last, int32_t* __restrict__ out_argmax,
                                         const uint32_t* __restrict__ emit_item) {
    const size_t HW = (size_t)width * height;
    const TileGeom<TILE, PPT, SPLIT> g(bin, part, ranges, tiles_x, tiles_per_view);
    bool inside[PPT];
    inside_mask(g, width, height, inside);
    float T[PPT], cr[PPT], cg[PPT], cb[PPT];
    uint32_t last[PPT], amax[PPT];
    bool masked;
    fwd_core<TILE, PPT, SPLIT, ARGMAX, DET>(g, inside, pval, emit_item, rec, kc, T, cr, cg, cb, last, amax, masked);
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        if (!inside[p]) continue;
        const size_t pix = (size_t)g.py(p) * width + g.px;
        out_rgb[(size_t)g.view * 3 * HW + pix] = cr[p];
        out_rgb[(size_t)g.view * 3 * HW + HW + pix] = cg[p];
        out_rgb[(size_t)g.view * 3 * HW + 2 * HW + pix] = cb[p];
        out_T[g.view * HW + pix] = T[p];
        out_last[g.view * HW + pix] = last[p];
        if (ARGMAX)
            out_argmax[g.view * HW + pix] = amax[p] == 0xFFFFFFFFu ? -1 : (int32_t)(amax[p] - (uint32_t)g.view * n);
    }
}

template <int TILE, int PPT, bool ARGMAX, bool DET>
__global__ void __launch_bounds__(Layout<TILE, PPT>::kThreads)
    k_raster_fwd(const uint2* __restrict__ ranges, const uint32_t* __restrict__ pval, const float4* __restrict__ rec,
                 int width, int height, int tiles_x, int tiles_per_view, int n, DevConst kc,
                 float* __restrict__ out_rgb, float* __restrict__ out_T, uint32_t* __restrict__ out_last,
                 int32_t* __restrict__ out_argmax, uint32_t* __restrict__ queue,
                 const uint32_t* __restrict__ order, const uint32_t* __restrict__ emit_item) {
    int bin, half;
    while (next_work(queue, order, bin, half)) {
        if constexpr (Layout<TILE, PPT>::kHalves) {
            if (half >= 0) {
                fwd_item<TILE, 1, 2, ARGMAX, DET>(bin, half, ranges, pval, rec, width, height, tiles_x,
                                                  tiles_per_view, n, kc, out_rgb, out_T, out_last, out_argmax,
                                                  emit_item);
                continue;
            }
        }
        fwd_item<TILE, PPT, 1, ARGMAX, DET>(bin, 0, ranges, pval, rec, width, height, tiles_x, tiles_per_view, n, kc,
                                            out_rgb, out_T, out_last, out_argmax, emit_item);
    }
}

// One work item's adjoint.
template <int TILE, int PPT, int SPLIT, bool DET>
__device__ __forceinline__ void bwd_item(int bin, int part, const uint2* __restrict__ ranges,
                                         const uint32_t* __restrict__ pval, const float4* __restrict__ rec, int width,
                                         int height, int tiles_x, int tiles_per_view, const DevConst& kc,
                                         const float* __restrict__ T_final, const uint32_t* __restrict__ n_last,
                                         const float* __restrict__ dLdC, float* __restrict__ grad2d,
                                         const uint32_t* __restrict__ emit_item, float* __restrict__ pairgrad) {
    const size_t HW = (size_t)width * height;
    const TileGeom<TILE, PPT, SPLIT> g(bin, part, ranges, tiles_x, tiles_per_view);
    float T[PPT], gr[PPT], gg[PPT], gb[PPT];
    uint32_t cnt[PPT];
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        T[p] = 1.f;
        gr[p] = gg[p] = gb[p] = 0.f;
        cnt[p] = 0;
        if (g.px < width && g.py(p) < height) {
            const size_t pix = (size_t)g.py(p) * width + g.px;
            T[p] = T_final[g.view * HW + pix];
            cnt[p] = n_last[g.view * HW + pix];
            gr[p] = dLdC[(size_t)g.view * 3 * HW + pix];
            gg[p] = dLdC[(size_t)g.view * 3 * HW + HW + pix];
            gb[p] = dLdC[(size_t)g.view * 3 * HW + 2 * HW + pix];
        }
    }
    bwd_core<TILE, PPT, SPLIT, DET>(g, pval, emit_item, rec, kc, T, cnt, gr, gg, gb, grad2d, pairgrad, -1, false,
                                    false);
}

template <int TILE, int PPT, bool DET>
__global__ void __launch_bounds__(Layout<TILE, PPT>::kThreads)
    k_raster_bwd(const uint2* __restrict__ ranges, const uint32_t* __restrict__ pval, const float4* __restrict__ rec,
                 int width, int height, int tiles_x, int tiles_per_view, DevConst kc,
                 const float* __restrict__ T_final, const uint32_t* __restrict__ n_last,
                 const float* __restrict__ dLdC, float* __restrict__ grad2d, uint32_t* __restrict__ queue,
                 const uint32_t* __restrict__ order, const uint32_t* __restrict__ emit_item,
                 float* __restrict__ pairgrad) {
    int bin, half;
    while (next_work(queue, order, bin, half)) {
        if constexpr (Layout<TILE, PPT>::kHalves) {
            if (half >= 0) {
                bwd_item<TILE, 1, 2, DET>(bin, half, ranges, pval, rec, width, height, tiles_x, tiles_per_view, kc,
                                          T_final, n_last, dLdC, grad2d, emit_item, pairgrad);
                continue;
            }
        }
        bwd_item<TILE, PPT, 1, DET>(bin, 0, ranges, pval, rec, width, height, tiles_x, tiles_per_view, kc, T_final,
                                    n_last, dLdC, grad2d, emit_item, pairgrad);
    }
}

// One work item of a mapping iteration: forward (Eq. 3), the L1 term of Eq. 10 and
// dL/dC = lambda sign(C - I) / 3HW for its pixels, then the adjoint, with final T, last
// index and dL/dC kept in registers. Writes the image; returns the thread's photometric sum.
template <int TILE, int PPT, int SPLIT, bool DET>
__device__ __forceinline__ float fused_item(int bin, int part, const uint2* __restrict__ ranges,
                                            const uint32_t* __restrict__ pval, const float4* __restrict__ rec,
                                            int width, int height, int tiles_x, int tiles_per_view,
                                            const DevConst& kc, const float* __restrict__ target, float scale,
                                            float* __restrict__ out_rgb, float* __restrict__ grad2d,
                                            const uint32_t* __restrict__ emit_item, float* __restrict__ pairgrad,
                                            float* __restrict__ tile_part) {
    const size_t HW = (size_t)width * height;
    const TileGeom<TILE, PPT, SPLIT> g(bin, part, ranges, tiles_x, tiles_per_view);
    bool inside[PPT];
    inside_mask(g, width, height, inside);
    float T[PPT], cr[PPT], cg[PPT], cb[PPT], gr[PPT], gg[PPT], gb[PPT];
    uint32_t last[PPT], amax[PPT];
    bool masked;   // the last staged batch (of a one-batch tile: the one the adjoint may reuse)
    const int staged = fwd_core<TILE, PPT, SPLIT, false, DET>(g, inside, pval, emit_item, rec, kc, T, cr, cg, cb, last,
                                                              amax, masked);
    float tl = 0.f;   // this thread's photometric sum over the item
#pragma unroll
    for (int p = 0; p < PPT; ++p) {
        gr[p] = gg[p] = gb[p] = 0.f;
        if (!inside[p]) {
            last[p] = 0;
            continue;
        }
        const size_t pix = (size_t)g.py(p) * width + g.px;
        const size_t o = (size_t)g.view * 3 * HW + pix;
        out_rgb[o] = cr[p];
        out_rgb[o + HW] = cg[p];
        out_rgb[o + 2 * HW] = cb[p];
        const float r0 = cr[p] - target[o], r1 = cg[p] - target[o + HW], r2 = cb[p] - target[o + 2 * HW];
        tl += (fabsf(r0) + fabsf(r1)) + fabsf(r2);
        gr[p] = scale * (float)((r0 > 0.f) - (r0 < 0.f));
        gg[p] = scale * (float)((r1 > 0.f) - (r1 < 0.f));
        gb[p] = scale * (float)((r2 > 0.f) - (r2 < 0.f));
    }
    if constexpr (DET) {
        // deterministic mode: each tile's sum on its own (fixed tree), whichever CTA took it
        __shared__ float tred[32];
        float ts = tl;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ts += __shfl_xor_sync(0xFFFFFFFFu, ts, o);
        if ((threadIdx.x & 31) == 0) tred[threadIdx.x >> 5] = ts;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += tred[w];
            tile_part[bin] = t * scale;
        }
        __syncthreads();
    }
    bwd_core<TILE, PPT, SPLIT, DET>(g, pval, emit_item, rec, kc, T, last, gr, gg, gb, grad2d, pairgrad,
                                    (DET || !Layout<TILE, PPT, SPLIT>::kReuseStaged) ? -1 : staged, true, masked);
    return tl;
}

// One mapping iteration's compositing for every (view, tile). Writes the image and one
// photometric partial sum per CTA.
template <int TILE, int PPT, bool DET>
__global__ void __launch_bounds__(Layout<TILE, PPT>::kThreads, Layout<TILE, PPT>::kMinBlocks)
    k_raster_fused(const uint2* __restrict__ ranges, const uint32_t* __restrict__ pval,
                   const float4* __restrict__ rec, int width, int height, int tiles_x, int tiles_per_view,
                   DevConst kc, const float* __restrict__ target, const float* const* __restrict__ target_slot,
                   float scale, float* __restrict__ out_rgb, float* __restrict__ grad2d, float* __restrict__ partials,
                   uint32_t* __restrict__ queue, const uint32_t* __restrict__ order,
                   const uint32_t* __restrict__ emit_item, float* __restrict__ pairgrad,
                   float* __restrict__ tile_part) {
    if (target_slot != nullptr) target = *target_slot;   // a replayed graph's per-call target
    int bin, half;
    float loss = 0.f;
    while (next_work(queue, order, bin, half)) {
        if constexpr (Layout<TILE, PPT>::kHalves) {
            if (half >= 0) {
                loss += fused_item<TILE, 1, 2, DET>(bin, half, ranges, pval, rec, width, height, tiles_x,
                                                    tiles_per_view, kc, target, scale, out_rgb, grad2d, emit_item,
                                                    pairgrad, tile_part);
                continue;
            }
        }
        loss += fused_item<TILE, PPT, 1, DET>(bin, 0, ranges, pval, rec, width, height, tiles_x, tiles_per_view, kc,
                                              target, scale, out_rgb, grad2d, emit_item, pairgrad, tile_part);
    }
    // per-CTA photometric partial (already scaled)
    __shared__ float red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        partials[blockIdx.x] = t * scale;
    }
}

// Algorithmic work of the last render, by replaying the forward traversal per
// pixel: out[0] += list entries the forward pass reaches (up to and including
// the stopping one), out[1] += pairs blended, out[2] += list entries the
// backward pass reaches (up to the last blended one).
template <int TILE>
__global__ void __launch_bounds__(TILE* TILE) k_count_work(const uint2* __restrict__ ranges,
                                                           const float4* __restrict__ rec,
                                                           const uint32_t* __restrict__ pval,
                                                           const uint32_t* __restrict__ emit_item, int width, int height,
                                                           int tiles_x, int tiles_per_view, DevConst kc,
                                                           unsigned long long* __restrict__ out) {
    const int bin = blockIdx.x;
    const int view = bin / tiles_per_view;
    const int t = bin - view * tiles_per_view;
    const int tyi = t / tiles_x, txi = t - tyi * tiles_x;
    const int lx = threadIdx.x % TILE, ly = threadIdx.x / TILE;
    const int px = txi * TILE + lx, py = tyi * TILE + ly;
    if (px >= width || py >= height) return;
    const float ox = (float)((txi * TILE) & ~31), oy = (float)((tyi * TILE) & ~31);
    const float fx = (float)px - ox, fy = (float)py - oy;
    const uint2 rg = ranges[bin];
    float T = 1.f;
    unsigned long long tested = 0, blended = 0, walked = 0;
    for (uint32_t j = rg.x; j < rg.y; ++j) {
        const uint32_t item = emit_item != nullptr ? emit_item[pval[j]] : pval[j];
        float4 a, q, c;
        stage_record(rec, item, ox, oy, kc.alpha_min, a, q, c);
        ++tested;
        const float dx = fx - a.x, dy = fy - a.y;
        if (fabsf(dx) > a.z || fabsf(dy) > a.w) continue;
        const float p2 = power2_dy(q.z, __fmul_rn(q.y, dx), __fmul_rn(__fmul_rn(q.x, dx), dx), dy);
        if (p2 < c.w) continue;
        const float alpha = fminf(kc.alpha_max, __fmul_rn(q.w, ex2_approx(p2)));
        const float Tn = __fmul_rn(T, 1.f - alpha);
        if (Tn < kc.T_min) break;
        T = Tn;
        ++blended;
        walked = j - rg.x + 1;
    }
    atomicAdd(out + 0, tested);
    atomicAdd(out + 1, blended);
    atomicAdd(out + 2, walked);
}

}  // namespace

cudaError_t launch_count_work(gs_ctx* c, const DevConst& k, unsigned long long* out, cudaStream_t s) {
    const int tpv = c->hcam[0].tiles_x * c->hcam[0].tiles_y;
    if (c->n_bins == 0) return cudaSuccess;
    ++c->launches;
    if (c->tile == 16)
        k_count_work<16><<<c->n_bins, 256, 0, s>>>(c->ranges, c->rec, c->pval[c->pair_buf], c->emit_item, c->width,
                                                   c->height, c->hcam[0].tiles_x, tpv, k, out);
    else
        k_count_work<8><<<c->n_bins, 64, 0, s>>>(c->ranges, c->rec, c->pval[c->pair_buf], c->emit_item, c->width,
                                                 c->height, c->hcam[0].tiles_x, tpv, k, out);
    return cudaGetLastError();
}

// resident CTAs of a kernel on the whole GPU (cached per kernel instantiation)
template <int KIND, int TILE, int PPT, typename K>
static int resident_grid(K kernel, int threads, int num_sms) {
    static int cached = 0;
    if (cached == 0) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
            per_sm = 1;
        cached = per_sm * num_sms;
    }
    return cached;
}

template <int TILE, int PPT, bool DET>
static void fwd_launch(gs_ctx* c, const DevConst& k, float* rgb, int32_t* argmax, cudaStream_t s, int tpv) {
    constexpr int NT = Layout<TILE, PPT>::kThreads, kParts = Layout<TILE, PPT>::kHalves ? 2 : 1;
    if (argmax) {
        const int grid =
            std::min(resident_grid<0 + 4 * DET, TILE, PPT>(k_raster_fwd<TILE, PPT, true, DET>, NT, c->num_sms),
                     kParts * c->n_bins);
        k_raster_fwd<TILE, PPT, true, DET><<<grid, NT, 0, s>>>(c->ranges, c->pval[c->pair_buf], c->rec, c->width, c->height,
                                                          c->hcam[0].tiles_x, tpv, c->n, k, rgb, c->T_final,
                                                          c->n_last, argmax, c->dcount + 6, c->work_order,
                                                          c->emit_item);
    } else {
        const int grid =
            std::min(resident_grid<1 + 4 * DET, TILE, PPT>(k_raster_fwd<TILE, PPT, false, DET>, NT, c->num_sms),
                     kParts * c->n_bins);
        k_raster_fwd<TILE, PPT, false, DET><<<grid, NT, 0, s>>>(c->ranges, c->pval[c->pair_buf], c->rec, c->width,
                                                           c->height, c->hcam[0].tiles_x, tpv, c->n, k, rgb,
                                                           c->T_final, c->n_last, nullptr, c->dcount + 6,
                                                           c->work_order, c->emit_item);
    }
}

template <int TILE, int PPT, bool DET>
static void bwd_launch(gs_ctx* c, const DevConst& k, const float* dLdC, cudaStream_t s, int tpv) {
    constexpr int NT = Layout<TILE, PPT>::kThreads, kParts = Layout<TILE, PPT>::kHalves ? 2 : 1;
    const int grid =
        std::min(resident_grid<2 + 4 * DET, TILE, PPT>(k_raster_bwd<TILE, PPT, DET>, NT, c->num_sms), kParts * c->n_bins);
    k_raster_bwd<TILE, PPT, DET><<<grid, NT, 0, s>>>(c->ranges, c->pval[c->pair_buf], c->rec, c->width, c->height,
                                                c->hcam[0].tiles_x, tpv, k, c->T_final, c->n_last, dLdC, c->grad2d,
                                                c->dcount + 7, c->work_order, c->emit_item,
                                                c->pairgrad);
}

template <int TILE, int PPT, bool DET>
static void fused_launch(gs_ctx* c, const DevConst& k, const float* target, const float* const* target_slot,
                         float* rgb, cudaStream_t s, int tpv, float* partials, int max_grid, int* grid_out) {
    constexpr int NT = Layout<TILE, PPT>::kThreads, kParts = Layout<TILE, PPT>::kHalves ? 2 : 1;
    const int grid = std::min(
        std::min(resident_grid<3 + 4 * DET, TILE, PPT>(k_raster_fused<TILE, PPT, DET>, NT, c->num_sms),
                 kParts * c->n_bins),
        max_grid);
    const float scale = k.lambda_color / (float)(3 * (size_t)c->width * c->height);
    k_raster_fused<TILE, PPT, DET><<<grid, NT, 0, s>>>(c->ranges, c->pval[c->pair_buf], c->rec, c->width, c->height,
                                                  c->hcam[0].tiles_x, tpv, k, target, target_slot, scale, rgb,
                                                  c->grad2d, partials,
                                                  c->dcount + 6, c->work_order, c->emit_item,
                                                  c->pairgrad, c->tile_part);
    *grid_out = grid;
}

// The deterministic mode has one layout (8-px tiles, 2 pixels per thread: one
// warp per tile); the default mode any of the five.
#define GS_DISPATCH(FN, ...)                                         \
    do {                                                             \
        if (c->cfg.deterministic) {                                  \
            FN<8, 2, true>(__VA_ARGS__);                             \
        } else if (c->tile == 16) {                                  \
            if (c->ppt == 1) FN<16, 1, false>(__VA_ARGS__);          \
            else if (c->ppt == 2) FN<16, 2, false>(__VA_ARGS__);     \
            else FN<16, 4, false>(__VA_ARGS__);                      \
        } else {                                                     \
            if (c->ppt == 1) FN<8, 1, false>(__VA_ARGS__);           \
            else FN<8, 2, false>(__VA_ARGS__);                       \
        }                                                            \
    } while (0)

cudaError_t launch_raster_forward(gs_ctx* c, const DevConst& k, float* rgb, int32_t* argmax, cudaStream_t s) {
    const int tpv = c->hcam[0].tiles_x * c->hcam[0].tiles_y;
    if (c->n_bins == 0) return cudaSuccess;
    // work queue (a mapping iteration zeroes it on its side stream)
    cudaError_t e = c->side_zeroed ? cudaSuccess : cudaMemsetAsync(c->dcount + 6, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    ++c->launches;
    GS_DISPATCH(fwd_launch, c, k, rgb, argmax, s, tpv);
    return cudaGetLastError();
}

cudaError_t launch_raster_backward(gs_ctx* c, const DevConst& k, const float* dLdC, cudaStream_t s) {
    const int tpv = c->hcam[0].tiles_x * c->hcam[0].tiles_y;
    if (c->n_bins == 0) return cudaSuccess;
    // work queue (a mapping iteration zeroes it on its side stream)
    cudaError_t e = c->side_zeroed ? cudaSuccess : cudaMemsetAsync(c->dcount + 7, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    ++c->launches;
    GS_DISPATCH(bwd_launch, c, k, dLdC, s, tpv);
    return cudaGetLastError();
}

cudaError_t launch_raster_fused(gs_ctx* c, const DevConst& k, const float* target, const float* const* target_slot,
                                float* rgb, float* partials, int max_grid, int* grid_out, cudaStream_t s) {
    const int tpv = c->hcam[0].tiles_x * c->hcam[0].tiles_y;
    *grid_out = 0;
    if (c->n_bins == 0) return cudaSuccess;
    // work queue (a mapping iteration zeroes it on its side stream)
    cudaError_t e = c->side_zeroed ? cudaSuccess : cudaMemsetAsync(c->dcount + 6, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    ++c->launches;
    GS_DISPATCH(fused_launch, c, k, target, target_slot, rgb, s, tpv, partials, max_grid, grid_out);
    return cudaGetLastError();
}

}  // namespace gs
