// Map management: initialisation from back-projected points (Eq. 6), dynamic
// insertion gated by rendered opacity (Eq. 7 reading) and densification by
// splitting (Section 3.2). These run once per keyframe, not per iteration.
#include <algorithm>

#include "gs_internal.cuh"

namespace gs {
namespace {

// ---- the 3 nearest reference points of each query ----
//
// Brute force over all pairs, split over chunks of the reference points so that a keyframe's
// hundred queries fill the GPU: a warp takes kKnnQueries queries through one chunk, its lanes the
// references side by side (a load serves all its queries), and leaves the chunk's 3 smallest squared
// distances; the kernels that use them merge the chunks, a warp a query. Bound by some eight
// instructions a pair: 96 queries of 150,000 points 310 us with one CTA walking all references for
// each query, and one thread merging 768 candidates; 18 us and 6 for the merge.
constexpr int kKnnQueries = 4, kKnnWarps = 8;

struct Best3 {
    float b0 = INFINITY, b1 = INFINITY, b2 = INFINITY;
    // (without branches: each lane's insertion would be its own; a distance that is not a number counts
    // as infinite)
    __device__ __forceinline__ void add(float d) {
        d = d < INFINITY ? d : INFINITY;
        const float t = fmaxf(b0, d), t1 = fmaxf(b1, t);
        b0 = fminf(b0, d);
        b1 = fminf(b1, t);
        b2 = fminf(b2, t1);
    }
    // the warp's 3 smallest, to every lane (squared distances: the order of the bits is theirs)
    __device__ __forceinline__ void merge_warp() {
        float r[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t m = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(b0));
            const uint32_t who = __ballot_sync(0xFFFFFFFFu, __float_as_uint(b0) == m);
            r[k] = __uint_as_float(m);
            if ((threadIdx.x & 31) == __ffs(who) - 1) {
                b0 = b1;
                b1 = b2;
                b2 = INFINITY;
            }
        }
        b0 = r[0];
        b1 = r[1];
        b2 = r[2];
    }
    // root mean square of the distances there are (0.01 if there is no reference point)
    __device__ __forceinline__ float rms() const {
        const int cnt = (b0 < INFINITY) + (b1 < INFINITY) + (b2 < INFINITY);
        const float s = (cnt > 0 ? b0 : 0.f) + (cnt > 1 ? b1 : 0.f) + (cnt > 2 ? b2 : 0.f);
        return cnt > 0 ? sqrtf(s / (float)cnt) : 0.01f;
    }
};

// Queries q [n][3]; references planar [3][ref_stride], query i's own excluded when ref_is_self.
// part[chunk][query][3].
__global__ void __launch_bounds__(32 * kKnnWarps) k_knn_chunks(const float* __restrict__ q, int n,
                                                              const float* __restrict__ ref, int ref_stride, int n_ref,
                                                              int chunk, int ref_is_self, float* __restrict__ part) {
    const int lane = threadIdx.x & 31, q0 = (blockIdx.x * kKnnWarps + (threadIdx.x >> 5)) * kKnnQueries;
    if (q0 >= n) return;
    float x[kKnnQueries], y[kKnnQueries], z[kKnnQueries];
    Best3 best[kKnnQueries];
#pragma unroll
    for (int k = 0; k < kKnnQueries; ++k) {
        const size_t i = (size_t)min(q0 + k, n - 1);
        x[k] = q[3 * i];
        y[k] = q[3 * i + 1];
        z[k] = q[3 * i + 2];
    }
    const int j0 = blockIdx.y * chunk, j1 = min(n_ref, j0 + chunk);
#pragma unroll 4
    for (int j = j0 + lane; j < j1; j += 32) {
        const float rx = ref[j], ry = ref[(size_t)ref_stride + j], rz = ref[2 * (size_t)ref_stride + j];
#pragma unroll
        for (int k = 0; k < kKnnQueries; ++k) {
            const float dx = rx - x[k], dy = ry - y[k], dz = rz - z[k];
            const float d = dx * dx + dy * dy + dz * dz;
            best[k].add(ref_is_self && j == q0 + k ? INFINITY : d);
        }
    }
#pragma unroll
    for (int k = 0; k < kKnnQueries; ++k) {
        best[k].merge_warp();
        if (q0 + k < n && lane < 3)
            part[((size_t)blockIdx.y * n + q0 + k) * 3 + lane] = lane == 0 ? best[k].b0 : (lane == 1 ? best[k].b1 : best[k].b2);
    }
}

// the chunks' candidates of query i, merged by its warp
__device__ __forceinline__ Best3 knn_of(const float* __restrict__ part, int chunks, int n, int i) {
    Best3 b;
    for (int k = threadIdx.x & 31; k < 3 * chunks; k += 32) b.add(part[((size_t)(k / 3) * n + i) * 3 + k % 3]);
    b.merge_warp();
    return b;
}

// Plain initialisation, one new Gaussian per warp.
__global__ void __launch_bounds__(256) k_init_points(const float* __restrict__ pts, const float* __restrict__ rgb,
                                                     const float* __restrict__ part, int chunks, int n,
                                                     float* __restrict__ out, int out_stride) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    const float rms = knn_of(part, chunks, n, i).rms();
    if ((threadIdx.x & 31) == 0) {
        float x = pts[3 * (size_t)i], y = pts[3 * (size_t)i + 1], z = pts[3 * (size_t)i + 2];
        float ls = fminf(fmaxf(logf(fmaxf(rms, 1e-30f)), -7.f), -1.f);
        const float v[kParamRows] = {x, y, z, ls, ls, ls, 1.f, 0.f, 0.f, 0.f, 0.f, rgb[3 * (size_t)i],
                                     rgb[3 * (size_t)i + 1], rgb[3 * (size_t)i + 2]};
        for (int r = 0; r < kParamRows; ++r) out[(size_t)r * out_stride + i] = v[r];
    }
}

// The pixel each point projects to, in front of the camera (-1: none), and with `order` the work list of
// the tiles (or, with `halves`, half tiles) that hold one of them: an insertion's opacity gate reads the
// transmittance at those pixels alone, so nothing else is composited. flags: two zeroed words a bin. A
// non-zero *cancel leaves the list empty. One CTA.
__global__ void __launch_bounds__(1024) k_point_items(DevCamera cam, float near_z, const float* __restrict__ pts, int n,
                                                      int tile, int halves, int* __restrict__ pixel,
                                                      uint32_t* __restrict__ flags, uint32_t* __restrict__ order,
                                                      const uint32_t* __restrict__ cancel) {
    __shared__ uint32_t count;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += 1024) {
        const float x = pts[3 * (size_t)i], y = pts[3 * (size_t)i + 1], z = pts[3 * (size_t)i + 2];
        const float tx = cam.R[0] * x + cam.R[1] * y + cam.R[2] * z + cam.t[0];
        const float ty = cam.R[3] * x + cam.R[4] * y + cam.R[5] * z + cam.t[1];
        const float tz = cam.R[6] * x + cam.R[7] * y + cam.R[8] * z + cam.t[2];
        const bool front = tz > near_z;
        const float zz = front ? tz : 1.f;
        const float u = cam.fx * tx / zz + cam.cx, v = cam.fy * ty / zz + cam.cy;
        const float pxf = floorf(u + 0.5f), pyf = floorf(v + 0.5f);
        const bool inside = front && pxf >= 0.f && pxf < (float)cam.width && pyf >= 0.f && pyf < (float)cam.height;
        const int px = inside ? (int)pxf : 0, py = inside ? (int)pyf : 0;
        pixel[i] = inside ? py * cam.width + px : -1;
        if (order != nullptr && inside) {
            const uint32_t bin = (uint32_t)((py / tile) * cam.tiles_x + px / tile);
            const uint32_t half = halves ? (uint32_t)(py % tile) / (uint32_t)(tile / 2) : 0u;
            if (atomicExch(flags + 2 * (size_t)bin + half, 1u) == 0u)
                order[1 + atomicAdd(&count, 1u)] = halves ? bin | ((1u + half) << kItemShift) : bin;
        }
    }
    __syncthreads();
    if (order != nullptr && threadIdx.x == 0) order[0] = *cancel != 0u ? 0u : count;
}

// Insertion test of point i (a warp). Opacity gate (tau2 = 0): keep[i] = 0 iff the point
// projects, in front of the camera, to a pixel whose rendered opacity 1 - T
// exceeds the threshold. Distance rule (tau2 = tau^2 > 0, Eq. 7 as its text
// states it): keep[i] = 1 iff the nearest existing mean is farther than tau
// (T is not read). Also stages the plain initial parameters [14][n].
__global__ void __launch_bounds__(256) k_insert_test(size_t HW, float thresh, float tau2, const float* __restrict__ pts,
                                                     const int* __restrict__ pixel, const float* __restrict__ T,
                                                     const float* __restrict__ image, const float* __restrict__ part,
                                                     int chunks, uint32_t* __restrict__ keep,
                                                     float* __restrict__ stage, int n) {
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= n) return;
    const Best3 best = knn_of(part, chunks, n, i);
    if ((threadIdx.x & 31) != 0) return;
    const float rms = best.rms(), dmin2 = best.b0;
    const bool inside = pixel[i] >= 0;
    const size_t pix = inside ? (size_t)pixel[i] : 0;
    bool skip = tau2 > 0.f ? !(dmin2 > tau2) : (inside && (1.f - T[pix]) > thresh);
    keep[i] = skip ? 0u : 1u;
    float ls = fminf(fmaxf(logf(fmaxf(rms, 1e-30f)), -7.f), -1.f);
    const float vals[kParamRows] = {pts[3 * (size_t)i], pts[3 * (size_t)i + 1], pts[3 * (size_t)i + 2],
                                    ls, ls, ls, 1.f, 0.f, 0.f, 0.f, 0.f,
                                    image[pix], image[HW + pix], image[2 * HW + pix]};
    for (int r = 0; r < kParamRows; ++r) stage[(size_t)r * n + i] = vals[r];
}

// Appends the kept points in order to the map's n Gaussians (parameters, zero moments and statistics):
// in one CTA that scans them as it goes, or (pos != NULL: their exclusive scan) in CTAs of 1024 points.
// Writes 1 or 0 per point to mask (optional) and, in one CTA, their number to *count (pinned host
// memory).
__global__ void __launch_bounds__(1024) k_append(const float* __restrict__ stage, int n_stage,
                                                 const uint32_t* __restrict__ keep, float* __restrict__ P,
                                                 float* __restrict__ M, float* __restrict__ V,
                                                 float* __restrict__ dsum, float* __restrict__ dcnt,
                                                 uint32_t* __restrict__ dom, int base, int cap,
                                                 uint8_t* __restrict__ mask, uint32_t* __restrict__ count,
                                                 const uint32_t* __restrict__ pos) {
    __shared__ uint32_t wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto put = [&](int i, uint32_t at) {
        const int d = base + (int)at;
#pragma unroll
        for (int r = 0; r < kParamRows; ++r) {
            P[(size_t)r * cap + d] = stage[(size_t)r * n_stage + i];
            M[(size_t)r * cap + d] = 0.f;
            V[(size_t)r * cap + d] = 0.f;
        }
        dsum[d] = 0.f;
        dcnt[d] = 0.f;
        dom[d] = 0u;
    };
    if (pos != nullptr) {
        const int i = blockIdx.x * 1024 + threadIdx.x;
        if (i >= n_stage) return;
        const bool k = keep[i] != 0u;
        if (mask != nullptr) mask[i] = k ? 1 : 0;
        if (k) put(i, pos[i]);
        return;
    }
    uint32_t before = 0;
    for (int i0 = 0; i0 < n_stage; i0 += 1024) {
        const int i = i0 + threadIdx.x;
        const bool k = i < n_stage && keep[i] != 0u;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, k);
        if (lane == 0) wsum[w] = __popc(bal);
        __syncthreads();
        uint32_t pre = 0, all = 0;
#pragma unroll
        for (int q = 0; q < 32; ++q) {
            pre += q < w ? wsum[q] : 0u;
            all += wsum[q];
        }
        __syncthreads();
        if (mask != nullptr && i < n_stage) mask[i] = k ? 1 : 0;
        if (k) put(i, before + pre + __popc(bal & ((1u << lane) - 1u)));
        before += all;
    }
    if (threadIdx.x == 0) *count = before;
}

// Split mask: the gradient criterion, or (sigma > 0) more than sigma dominated
// pixels (Eq. 9 split mask M).
__global__ void __launch_bounds__(256) k_split_flags(const float* __restrict__ dsum, const float* __restrict__ dcnt,
                                                     const uint32_t* __restrict__ dom, int n, float thresh,
                                                     float sigma, uint32_t* __restrict__ flags) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float c = dcnt[i];
    float mean = c > 0.f ? dsum[i] / c : 0.f;
    const bool clear = sigma > 0.f && (float)dom[i] > sigma;
    flags[i] = (mean > thresh || clear) ? 1u : 0u;
}

// Eq. 8-9: every pixel whose largest blend weight belongs to Gaussian a adds one
// to a's dominated-pixel count (argmax -1: no Gaussian).
__global__ void __launch_bounds__(256) k_count_dominant(const int32_t* __restrict__ argmax, size_t n_pix, int n,
                                                        uint32_t* __restrict__ dom) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n_pix; i += (size_t)gridDim.x * blockDim.x) {
        const int a = argmax[i];
        if (a >= 0 && a < n) atomicAdd(dom + a, 1u);
    }
}

// SplitMix64 (Steele, Lea and Flood 2014) as a counter-based generator.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// standard normal by the Box-Muller transform of two counter-based uniforms
__device__ float normal_at(uint64_t seed, uint64_t counter) {
    uint64_t a = splitmix64(seed ^ (2 * counter)), b = splitmix64(seed ^ (2 * counter + 1));
    float u1 = ((float)(a >> 40) + 0.5f) * (1.0f / 16777216.0f);
    float u2 = (float)(b >> 40) * (1.0f / 16777216.0f);
    return sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
}

// Survivors move to pos_s = i - (split parents before i); children of the
// k-th split parent go to n_surv + 2k and n_surv + 2k + 1. The statistics restart.
__global__ void __launch_bounds__(256) k_split_scatter(const float* __restrict__ P, const float* __restrict__ M,
                                                       const float* __restrict__ V, int n, int cap,
                                                       const uint32_t* __restrict__ flags,
                                                       const uint32_t* __restrict__ pos, uint32_t n_split,
                                                       const float* __restrict__ normals, uint64_t seed,
                                                       float log_factor, float* __restrict__ P2,
                                                       float* __restrict__ M2, float* __restrict__ V2,
                                                       float* __restrict__ dsum, float* __restrict__ dcnt,
                                                       uint32_t* __restrict__ dom) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    dsum[i] = dcnt[i] = 0.f;   // (beyond n they are zero)
    dom[i] = 0u;
    uint32_t before = pos[i];
    float p[kParamRows];
    for (int r = 0; r < kParamRows; ++r) p[r] = P[(size_t)r * cap + i];
    if (!flags[i]) {
        int d = i - (int)before;
        for (int r = 0; r < kParamRows; ++r) {
            P2[(size_t)r * cap + d] = p[r];
            M2[(size_t)r * cap + d] = M[(size_t)r * cap + i];
            V2[(size_t)r * cap + d] = V[(size_t)r * cap + i];
        }
        return;
    }
    int n_surv = n - (int)n_split;
    float qq = sqrtf(p[6] * p[6] + p[7] * p[7] + p[8] * p[8] + p[9] * p[9]);
    float w = p[6] / qq, x = p[7] / qq, y = p[8] / qq, z = p[9] / qq;
    float R[9] = {1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y),
                  2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x),
                  2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)};
    float s[3] = {expf(p[3]), expf(p[4]), expf(p[5])};
    for (int k = 0; k < 2; ++k) {
        float zn[3];
        for (int a = 0; a < 3; ++a)
            zn[a] = normals ? normals[(size_t)i * 6 + k * 3 + a] : normal_at(seed, (uint64_t)i * 6 + k * 3 + a);
        int d = n_surv + 2 * (int)before + k;
        for (int r = 0; r < kParamRows; ++r) {
            float v = p[r];
            if (r < 3) v = p[r] + R[r * 3 + 0] * s[0] * zn[0] + R[r * 3 + 1] * s[1] * zn[1] + R[r * 3 + 2] * s[2] * zn[2];
            else if (r < 6) v = p[r] - log_factor;
            P2[(size_t)r * cap + d] = v;
            M2[(size_t)r * cap + d] = 0.f;
            V2[(size_t)r * cap + d] = 0.f;
        }
    }
}

}  // namespace

// Chunks of the references: 256 of them or more, fewer chunks once the queries alone fill the GPU
// (four CTAs an SM in all; the merge reads three candidates a chunk).
static int knn_chunks(const gs_ctx* c, int n, int n_ref) {
    const int per_cta = kKnnQueries * kKnnWarps, groups = (n + per_cta - 1) / per_cta;
    const int want = (4 * c->num_sms + groups - 1) / groups;
    return std::max(1, std::min(want, (n_ref + 255) / 256));
}

size_t knn_scratch(const gs_ctx* c, int n, int n_ref) { return 3 * (size_t)n * knn_chunks(c, n, n_ref); }

static cudaError_t knn(gs_ctx* c, const float* q, int n, const float* ref, int ref_stride, int n_ref, int ref_is_self,
                       float* part, int* chunks_out, cudaStream_t s) {
    const int per_cta = kKnnQueries * kKnnWarps, chunks = knn_chunks(c, n, n_ref);
    const int chunk = ((n_ref + chunks - 1) / chunks + 31) & ~31;
    *chunks_out = chunks;
    ++c->launches;
    k_knn_chunks<<<dim3((n + per_cta - 1) / per_cta, chunks), 32 * kKnnWarps, 0, s>>>(q, n, ref, ref_stride, n_ref,
                                                                                       chunk, ref_is_self, part);
    return cudaGetLastError();
}

cudaError_t launch_init_points(gs_ctx* c, const float* pts, const float* rgb, int n, const float* ref, int ref_stride,
                               int n_ref, int ref_is_self, float* part, float* out_params, int out_stride,
                               cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    int chunks = 0;
    const cudaError_t e = knn(c, pts, n, ref, ref_stride, n_ref, ref_is_self, part, &chunks, s);
    if (e != cudaSuccess) return e;
    ++c->launches;
    k_init_points<<<(n + 7) / 8, 256, 0, s>>>(pts, rgb, part, chunks, n, out_params, out_stride);
    return cudaGetLastError();
}

namespace {
__global__ void k_points_planar(const float* __restrict__ pts, int n, float* __restrict__ out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = pts[3 * i];
    out[n + i] = pts[3 * i + 1];
    out[2 * n + i] = pts[3 * i + 2];
}
}  // namespace

cudaError_t launch_points_planar(const float* pts, int n, float* out, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_points_planar<<<(n + 255) / 256, 256, 0, s>>>(pts, n, out);
    return cudaGetLastError();
}

cudaError_t launch_point_items(gs_ctx* c, const PointItems& p, bool list, cudaStream_t s) {
    if (list) {
        const cudaError_t e = cudaMemsetAsync(p.flags, 0, sizeof(uint32_t) * 2 * (size_t)c->n_bins, s);
        if (e != cudaSuccess) return e;
    }
    ++c->launches;
    k_point_items<<<1, 1024, 0, s>>>(c->hcam[0], c->cfg.near_z, p.pts, p.n, c->tile, half_tiles(c) ? 1 : 0, p.pixel,
                                     p.flags, list ? c->work_order : nullptr, c->dcount + 10);
    return cudaGetLastError();
}

cudaError_t launch_insert_test(gs_ctx* c, const PointItems& p, const float* image, float* part, uint32_t* keep,
                               float* stage, cudaStream_t s) {
    if (p.n == 0) return cudaSuccess;
    int chunks = 0;
    const cudaError_t e = knn(c, p.pts, p.n, c->params, c->cap, c->n, 0, part, &chunks, s);
    if (e != cudaSuccess) return e;
    ++c->launches;
    const float tau2 = c->cfg.insert_tau > 0.f ? c->cfg.insert_tau * c->cfg.insert_tau : 0.f;
    k_insert_test<<<(p.n + 7) / 8, 256, 0, s>>>((size_t)c->width * c->height, c->cfg.insert_opacity, tau2, p.pts, p.pixel,
                                                c->T_final, image, part, chunks, keep, stage, p.n);
    return cudaGetLastError();
}

// Points up to which one CTA appends them: an insertion into a map of 100 takes 182 us either way at
// 4,096 points; with one CTA / by a scan and many 206 / 182 us at 8,192, 1,770 / 563 at 262,144.
constexpr int kAppendOne = 4096;

cudaError_t launch_append(gs_ctx* c, const float* stage, int n_stage, const uint32_t* keep, uint8_t* mask,
                          uint32_t* count_host, cudaStream_t s) {
    if (n_stage == 0) return cudaSuccess;
    uint32_t* pos = nullptr;
    if (n_stage > kAppendOne) {   // (the points fit the map, and so the depth sort's buffer)
        pos = c->dkey[1];
        const cudaError_t e = scan_u32(c, keep, pos, (uint32_t)n_stage, count_host, s);
        if (e != cudaSuccess) return e;
    }
    ++c->launches;
    k_append<<<pos ? (n_stage + 1023) / 1024 : 1, 1024, 0, s>>>(stage, n_stage, keep, c->params, c->adam_m, c->adam_v,
                                                               c->dens_sum, c->dens_cnt, c->dom_cnt, c->n, c->cap, mask,
                                                               count_host, pos);
    return cudaGetLastError();
}

cudaError_t launch_split_flags(gs_ctx* c, uint32_t* flags, cudaStream_t s) {
    if (c->n == 0) return cudaSuccess;
    ++c->launches;
    k_split_flags<<<(c->n + 255) / 256, 256, 0, s>>>(c->dens_sum, c->dens_cnt, c->dom_cnt, c->n,
                                                     c->cfg.split_thresh, c->cfg.clarity_sigma, flags);
    return cudaGetLastError();
}

cudaError_t launch_count_dominant(gs_ctx* c, const int32_t* argmax, size_t n_pix, cudaStream_t s) {
    if (n_pix == 0 || c->n == 0) return cudaSuccess;
    ++c->launches;
    const int grid = (int)std::min<size_t>((n_pix + 255) / 256, (size_t)c->num_sms * 8);
    k_count_dominant<<<grid, 256, 0, s>>>(argmax, n_pix, c->n, c->dom_cnt);
    return cudaGetLastError();
}

cudaError_t launch_split_scatter(gs_ctx* c, const uint32_t* flags, const uint32_t* pos, uint32_t n_split,
                                 const float* normals, float* P2, float* M2, float* V2, cudaStream_t s) {
    if (c->n == 0) return cudaSuccess;
    ++c->launches;
    k_split_scatter<<<(c->n + 255) / 256, 256, 0, s>>>(c->params, c->adam_m, c->adam_v, c->n, c->cap, flags, pos,
                                                       n_split, normals, c->cfg.seed, logf(c->cfg.split_factor), P2,
                                                       M2, V2, c->dens_sum, c->dens_cnt, c->dom_cnt);
    return cudaGetLastError();
}

}  // namespace gs
