// The learned initialiser: a 3-layer MLP 80 -> 128 -> 128 -> 16 (11 used) with
// GELU, on the tensor cores in BF16 with FP32 accumulation, with hand-written
// forward, backward (MSE against converged Gaussian parameters) and Adam. It
// predicts log-scale (3), quaternion (4), opacity logit (1) and colour (3) of
// a Gaussian inserted at a VO point from the keyframe's 5x5 patch around the
// point, its depth and its camera-frame position.
//
// A CTA takes 32 or 64 rows through the whole network (and, in training, back through it) in one launch,
// on tcgen05.mma with bf16 operands in shared memory and f32 accumulators in TMEM. Upstream
// gradients dZ enter as bf16 hi + lo pairs (two products), so the backward
// keeps ~16 mantissa bits where one bf16 rounding would keep 8.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kIn = 80, kHid = 128, kOut = 11, kOutPad = 16;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kHid * kIn, kOffW2 = kOffB1 + kHid, kOffB2 = kOffW2 + kHid * kHid,
              kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kOutPad * kHid, kParams = kOffB3 + kOutPad;

typedef __nv_bfloat16 bf16;

constexpr uint32_t kTcWaitLimit = 1u << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// tcgen05 shared-memory matrix descriptor: start address, leading and stride
// byte offsets (all >> 4), the fixed version bits 46..48 = 0b001, no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// instruction descriptor of kind::f16: D = F32 (bits 4..5), A = B = BF16 (bits 7..9,
// 10..12), both K-major (bits 15, 16 clear), N >> 3 in bits 17..22, M >> 4 in 24..28
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit = kTcWaitLimit) {
    for (uint32_t i = 0; i < limit; ++i) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }

__device__ __forceinline__ float gelu_grad_f(float x) {
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// v = hi + lo with hi = bf16(v), lo = bf16(v - hi): a bf16 pair carrying ~16 mantissa bits
__device__ __forceinline__ void split_bf16(float v, bf16& hi, bf16& lo) {
    hi = __float2bfloat16_rn(v);
    lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// ---- operands in shared memory ----
//
// Canonical K-major, non-swizzled UMMA layout of a (rows x K) bf16 operand: 8 x 16-byte core
// matrices, the core of row group g and K group j at (g K / 8 + j) * 128 bytes: the leading (K)
// byte offset is 128, the stride (row-group) byte offset 16 K.
template <int K>
__host__ __device__ __forceinline__ constexpr uint32_t core_off(int row, int k) {
    return (uint32_t)((row >> 3) * (K * 16) + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

constexpr int kNetThreads = 256;     // 8 warps: 4 over the 128 TMEM lanes, twice over the rows of a pass

// The bf16 weights as the kernels copy them into shared memory, already in that layout (byte
// offsets): W1, W2, W3, then the transposes the input gradients need.
constexpr uint32_t kImgW1 = 0, kImgW2 = kImgW1 + kHid * kIn * 2, kImgW3 = kImgW2 + kHid * kHid * 2,
                   kImgW2T = kImgW3 + kOutPad * kHid * 2, kImgW3T = kImgW2T + kHid * kHid * 2,
                   kImgBytes = kImgW3T + kHid * kOutPad * 2, kImgForward = kImgW2T;

// Shared memory (byte offsets). The product with W3 takes 128 operand rows of which 16 exist: it
// reads 28 KB past W3, whatever lies there, into accumulator lanes nobody reads. H1 and H2 (rows x
// hidden) are dead once Z2 and Y are formed; dZ2 (rows x hidden, hi and lo) takes their place, and
// then dZ1^T.
constexpr uint32_t kSmW = 0;                                   // the weight image
template <bool TRAIN, int ROWS>
struct Smem {
    static constexpr uint32_t X = TRAIN ? kImgBytes : kImgForward;                // [row][in]
    static constexpr uint32_t H1 = X + ROWS * kIn * 2;                           // [row][hid]
    static constexpr uint32_t H2 = H1 + ROWS * kHid * 2;                         // [row][hid]
    static constexpr uint32_t Bias = H2 + ROWS * kHid * 2;                       // b1, b2, b3 (f32)
    static constexpr uint32_t ForwardEnd = Bias + (2 * kHid + kOutPad) * 4;
    // training only
    static constexpr uint32_t XT = (ForwardEnd + 127) / 128 * 128;                // [in][row]
    static constexpr uint32_t H1T = XT + kIn * ROWS * 2;                         // [hid][row]
    static constexpr uint32_t H2T = H1T + kHid * ROWS * 2;                       // [hid][row]
    static constexpr uint32_t DY = H2T + kHid * ROWS * 2;                        // [row][out], hi then lo
    static constexpr uint32_t DYT = DY + 2 * ROWS * kOutPad * 2;                 // [out][row], hi then lo
    static constexpr uint32_t DZT = DYT + 2 * ROWS * kOutPad * 2;                // [hid][row], hi then lo
    static constexpr uint32_t Target = DZT + 2 * kHid * ROWS * 2;                // [row][16] f32
    static constexpr uint32_t DZ = H1;                                            // [row][hid], hi then lo
    static constexpr uint32_t Past3 = kImgW3 + 128 * kHid * 2;                    // read by the product with W3
    static constexpr uint32_t Bytes = TRAIN ? Target + ROWS * kOutPad * 4 : (ForwardEnd > Past3 ? ForwardEnd : Past3);
};
static_assert(Smem<true, 64>::Bytes <= 227 * 1024, "shared memory of the training kernel");
static_assert(Smem<true, 32>::Past3 <= Smem<true, 32>::Bytes, "the product with W3 reads within shared memory");

// TMEM columns (f32 accumulators): Z1, Z2, Y and an input gradient, hidden (output) x rows; the
// weight gradients dW2, dW1 and dW3^T, summed over the CTA's passes.
constexpr uint32_t kTmZ1 = 0, kTmZ2 = 64, kTmY = 128, kTmDH = 192, kTmW2 = 256, kTmW1 = 384, kTmW3T = 464;

// D (128 x N, TMEM) (+)= A (128 x K) B (N x K)^T; one thread issues it.
template <int K, int N>
__device__ __forceinline__ void umma(uint32_t d, uint32_t a, uint32_t b, bool accumulate) {
    constexpr uint32_t idesc = umma_idesc_bf16(128, N);
#pragma unroll
    for (int kk = 0; kk < K / 16; ++kk) {
        const uint64_t ad = umma_desc(a + kk * 256, 128, K * 16);
        const uint64_t bd = umma_desc(b + kk * 256, 128, K * 16);
        const uint32_t acc = (accumulate || kk > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
            : "memory");
    }
}

// 16 consecutive accumulator columns of the thread's TMEM lane (the load is not waited for)
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float* f) {
    uint32_t v[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(addr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) f[i] = __uint_as_float(v[i]);
}
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t addr, float (&f)[N]) {
#pragma unroll
    for (int i = 0; i < N; i += 16) tmem_ld16(addr + i, f + i);
}

// N values of one operand row, columns r0 .. r0 + N - 1, as bf16 into [row][ROWS]
template <int ROWS, int N>
__device__ __forceinline__ void store_row(uint8_t* dst, int row, int r0, const bf16 (&h)[N]) {
#pragma unroll
    for (int g = 0; g < N; g += 8)
        *reinterpret_cast<uint4*>(dst + core_off<ROWS>(row, r0 + g)) = *reinterpret_cast<const uint4*>(h + g);
}
// the same values as one column (hidden unit j) of [row][kHid]
template <int N>
__device__ __forceinline__ void store_col(uint8_t* dst, int r0, int j, const bf16 (&h)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) *reinterpret_cast<bf16*>(dst + core_off<kHid>(r0 + i, j)) = h[i];
}

// The network over passes of ROWS rows, and in training its adjoint: forward, MSE over the 11
// outputs, dY = 2 (Y - T) / (n 11), and the gradient of every parameter, as this CTA's partial sums
// part[blockIdx.x][kParams], with its loss in loss_part.
//
// Every product has the 128 hidden units as its M dimension and rows (or units) as N, so a small
// batch spreads over SMs and no accumulator lane is padding; a thread owns one hidden unit and half of
// a pass's rows. What bounds it is latency: eight products, each a few hundred tensor cycles, and between
// them a read of TMEM, an erf (and, back, an exp) a value and a rewrite of the operands. With k_mlp_reduce
// it takes the place of 21 launches (elementwise kernels and strided GEMMs that gathered their operands
// element by element; 7 of them for a prediction alone): gradients of 4,096 rows 400 -> 20 us, a
// prediction of 96 rows 58 -> 6 us.
//
// A wait that gives up ends the CTA's work: it writes nothing, sets both flags of `err`, and leaves once
// its weight copy and its products have ended (a bounded wait again), so that neither runs on in shared
// memory or TMEM that is no longer its own.
struct NetErr {
    uint32_t* device;     // read by the kernels that would use the results
    uint32_t* host;       // pinned: read by the next calls
    uint32_t give_up;     // tests: the wait of each CTA (counted from 1) that gives up at once; 0: none
};
template <bool TRAIN, int ROWS>
__global__ void __launch_bounds__(kNetThreads, 1)
    k_mlp_net(const float* __restrict__ feat, const float* __restrict__ tgt, int n, const uint8_t* __restrict__ img,
              const float* __restrict__ par, float* __restrict__ out, float* __restrict__ part,
              float* __restrict__ loss_part, NetErr err) {
    typedef Smem<TRAIN, ROWS> S;
    constexpr int N = ROWS / 2;                  // rows of a thread
    extern __shared__ __align__(1024) uint8_t sm[];
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ uint32_t tmem_slot;
    __shared__ float red[2][kHid];
    constexpr uint32_t kCols = TRAIN ? 512u : 256u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = (warp & 3) * 32 + lane;        // hidden unit (output of the last layer)
    const int r0 = (warp >> 2) * N;              // first of the thread's rows of the pass
    const uint32_t base = smem_u32(sm), wbar = smem_u32(&bars[0]), bar = smem_u32(&bars[1]);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(wbar) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        constexpr uint32_t bytes = TRAIN ? kImgBytes : kImgForward;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(wbar), "r"(bytes) : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(base + kSmW),
            "l"(img), "r"(bytes), "r"(wbar)
            : "memory");
    }
    float* bias = reinterpret_cast<float*>(sm + S::Bias);
    for (int i = threadIdx.x; i < 2 * kHid + kOutPad; i += kNetThreads)
        bias[i] = par[i < kHid ? kOffB1 + i : (i < 2 * kHid ? kOffB2 + i - kHid : kOffB3 + i - 2 * kHid)];
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float b1 = bias[j], b2 = bias[kHid + j];
    uint32_t parity = 0, waits = 0;
    bool ok = true, weights_in = false, products_in = true;
    auto wait = [&](uint32_t b, uint32_t par) {
        return __syncthreads_and(mbar_wait(b, par, ++waits == err.give_up ? 0u : kTcWaitLimit)) != 0;
    };
    // the operands written so far become visible to the tensor cores, one thread issues, all wait
    auto products = [&](auto issue) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            issue();
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                         : "memory");
        }
        ok = products_in = wait(bar, parity);
        parity ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        return ok;
    };
    float db1 = 0.f, db2 = 0.f, db3 = 0.f, loss = 0.f;
    const float scale = 2.f / ((float)n * (float)kOut);
    bool first = true;
    const bool feat_vec = (reinterpret_cast<uintptr_t>(feat) & 15) == 0;
    const int passes = (n + ROWS - 1) / ROWS;
    for (int pass = blockIdx.x; pass < passes && ok; pass += gridDim.x) {
        const int row0 = pass * ROWS;
        for (int e = threadIdx.x; e < ROWS * (kIn / 8); e += kNetThreads) {
            const int g = e / ROWS, r = e - g * ROWS;
            __align__(16) bf16 h[8];
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (row0 + r < n) {
                const float* src = feat + (size_t)(row0 + r) * kIn + 8 * g;
                if (feat_vec) {
                    a = *reinterpret_cast<const float4*>(src);
                    b = *reinterpret_cast<const float4*>(src + 4);
                } else {
                    a = make_float4(src[0], src[1], src[2], src[3]);
                    b = make_float4(src[4], src[5], src[6], src[7]);
                }
            }
            const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int q = 0; q < 8; ++q) h[q] = __float2bfloat16_rn(x[q]);
            *reinterpret_cast<uint4*>(sm + S::X + core_off<kIn>(r, 8 * g)) = *reinterpret_cast<const uint4*>(h);
            if constexpr (TRAIN) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    *reinterpret_cast<bf16*>(sm + S::XT + core_off<ROWS>(8 * g + q, r)) = h[q];
            }
        }
        if constexpr (TRAIN) {
            float* st = reinterpret_cast<float*>(sm + S::Target);
            for (int e = threadIdx.x; e < ROWS * kOutPad; e += kNetThreads)
                st[e] = row0 + e / kOutPad < n ? tgt[(size_t)row0 * kOutPad + e] : 0.f;
        }
        if (first && !(ok = weights_in = wait(wbar, 0))) break;   // the weights have arrived
        float z[N];
        __align__(16) bf16 h[N];
        if (!products([&] { umma<kIn, ROWS>(tmem + kTmZ1, base + kSmW + kImgW1, base + S::X, false); })) break;
        tmem_ld(tlane + kTmZ1 + r0, z);
#pragma unroll
        for (int i = 0; i < N; ++i) h[i] = __float2bfloat16_rn(gelu_f(z[i] + b1));
        store_col(sm + S::H1, r0, j, h);
        if constexpr (TRAIN) store_row<ROWS>(sm + S::H1T, j, r0, h);
        if (!products([&] { umma<kHid, ROWS>(tmem + kTmZ2, base + kSmW + kImgW2, base + S::H1, false); })) break;
        tmem_ld(tlane + kTmZ2 + r0, z);
#pragma unroll
        for (int i = 0; i < N; ++i) h[i] = __float2bfloat16_rn(gelu_f(z[i] + b2));
        store_col(sm + S::H2, r0, j, h);
        if constexpr (TRAIN) store_row<ROWS>(sm + S::H2T, j, r0, h);
        if (!products([&] { umma<kHid, ROWS>(tmem + kTmY, base + kSmW + kImgW3, base + S::H2, false); })) break;
        if ((warp & 3) == 0) {   // outputs: lanes 0 .. 15
            tmem_ld(tlane + kTmY + r0, z);
            if (lane < kOutPad) {
                const float b3 = bias[2 * kHid + lane];
                if constexpr (!TRAIN) {
                    for (int i = 0; i < N; ++i)
                        if (row0 + r0 + i < n) out[(size_t)(row0 + r0 + i) * kOutPad + lane] = z[i] + b3;
                } else {
                    const float* st = reinterpret_cast<const float*>(sm + S::Target);
#pragma unroll
                    for (int i = 0; i < N; ++i) {
                        const int r = r0 + i;
                        float g = 0.f;
                        if (lane < kOut && row0 + r < n) {
                            const float d = z[i] + b3 - st[r * kOutPad + lane];
                            loss += d * d;
                            g = scale * d;
                            db3 += g;
                        }
                        bf16 hi, lo;
                        split_bf16(g, hi, lo);
                        *reinterpret_cast<bf16*>(sm + S::DY + core_off<kOutPad>(r, lane)) = hi;
                        *reinterpret_cast<bf16*>(sm + S::DY + ROWS * kOutPad * 2 + core_off<kOutPad>(r, lane)) = lo;
                        *reinterpret_cast<bf16*>(sm + S::DYT + core_off<ROWS>(lane, r)) = hi;
                        *reinterpret_cast<bf16*>(sm + S::DYT + ROWS * kOutPad * 2 + core_off<ROWS>(lane, r)) = lo;
                    }
                }
            }
        }
        if constexpr (TRAIN) {
            constexpr uint32_t dyl = ROWS * kOutPad * 2, dzl = ROWS * kHid * 2;
            // dH2 = dY W3 and dW3 = dY^T H2, both transposed
            if (!products([&] {
                    umma<kOutPad, ROWS>(tmem + kTmDH, base + kSmW + kImgW3T, base + S::DY, false);
                    umma<kOutPad, ROWS>(tmem + kTmDH, base + kSmW + kImgW3T, base + S::DY + dyl, true);
                    umma<ROWS, kOutPad>(tmem + kTmW3T, base + S::H2T, base + S::DYT, !first);
                    umma<ROWS, kOutPad>(tmem + kTmW3T, base + S::H2T, base + S::DYT + dyl, true);
                }))
                break;
            __align__(16) bf16 l[N];
            float dh[N];
            tmem_ld(tlane + kTmDH + r0, dh);
            tmem_ld(tlane + kTmZ2 + r0, z);
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const float v = dh[i] * gelu_grad_f(z[i] + b2);
                db2 += v;
                split_bf16(v, h[i], l[i]);
            }
            store_row<ROWS>(sm + S::DZT, j, r0, h);
            store_row<ROWS>(sm + S::DZT + dzl, j, r0, l);
            store_col(sm + S::DZ, r0, j, h);
            store_col(sm + S::DZ + dzl, r0, j, l);
            // dH1^T = W2^T dZ2^T and dW2 = dZ2^T H1
            if (!products([&] {
                    umma<kHid, ROWS>(tmem + kTmDH, base + kSmW + kImgW2T, base + S::DZ, false);
                    umma<kHid, ROWS>(tmem + kTmDH, base + kSmW + kImgW2T, base + S::DZ + dzl, true);
                    umma<ROWS, kHid>(tmem + kTmW2, base + S::DZT, base + S::H1T, !first);
                    umma<ROWS, kHid>(tmem + kTmW2, base + S::DZT + dzl, base + S::H1T, true);
                }))
                break;
            tmem_ld(tlane + kTmDH + r0, dh);
            tmem_ld(tlane + kTmZ1 + r0, z);
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const float v = dh[i] * gelu_grad_f(z[i] + b1);
                db1 += v;
                split_bf16(v, h[i], l[i]);
            }
            store_row<ROWS>(sm + S::DZ, j, r0, h);
            store_row<ROWS>(sm + S::DZ + dzl, j, r0, l);
            // dW1 = dZ1^T X
            if (!products([&] {
                    umma<ROWS, kIn>(tmem + kTmW1, base + S::DZ, base + S::XT, !first);
                    umma<ROWS, kIn>(tmem + kTmW1, base + S::DZ + dzl, base + S::XT, true);
                }))
                break;
        } else {
            __syncthreads();
        }
        first = false;
    }
    if (!ok) {
        if (!weights_in) mbar_wait(wbar, 0);
        if (!products_in) mbar_wait(bar, parity ^ 1u);
        if (threadIdx.x == 0) *err.device = *err.host = 1u;
    } else if constexpr (TRAIN) {
        float* P = part + (size_t)blockIdx.x * kParams;
        const int half = warp >> 2;
        float f[32];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int i0 = half * 64 + c * 32;
            tmem_ld(tlane + kTmW2 + i0, f);
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4*>(P + kOffW2 + j * kHid + i0 + i) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
        }
        {   // dW1: 80 columns, 48 and 32 of them a half
            tmem_ld(tlane + kTmW1 + half * 48, f);
#pragma unroll
            for (int i = 0; i < 32; i += 4)
                *reinterpret_cast<float4*>(P + kOffW1 + j * kIn + half * 48 + i) =
                    make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
            float e[16];
            tmem_ld(tlane + (half == 0 ? kTmW1 + 32 : kTmW3T), e);
            if (half == 0) {
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *reinterpret_cast<float4*>(P + kOffW1 + j * kIn + 32 + i) =
                        make_float4(e[i], e[i + 1], e[i + 2], e[i + 3]);
            } else {
                // the padding rows of the output layer are not trained
#pragma unroll
                for (int o = 0; o < kOutPad; ++o) P[kOffW3 + o * kHid + j] = o < kOut ? e[o] : 0.f;
            }
        }
        // the two row halves' bias gradients and losses
        if (half == 1) {
            red[0][j] = db1;
            red[1][j] = db2;
        }
        __syncthreads();
        if (half == 0) {
            P[kOffB1 + j] = db1 + red[0][j];
            P[kOffB2 + j] = db2 + red[1][j];
        }
        __syncthreads();
        if (warp == 4 && lane < kOutPad) {
            red[0][lane] = db3;
            red[1][lane] = loss;
        }
        __syncthreads();
        if (warp == 0) {
            float t = lane < kOutPad ? loss + red[1][lane] : 0.f;
            if (lane < kOutPad) P[kOffB3 + lane] = db3 + red[0][lane];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
            if (lane == 0) loss_part[blockIdx.x] = t / ((float)n * (float)kOut);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

// The CTAs' partial gradients and losses, added in a fixed order (so a step repeats bit for bit):
// 32 groups of four parameters a CTA, eight threads a group. Bound by its one read of the partials
// (113 KB a CTA of k_mlp_net, from L2).
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ part, const float* __restrict__ loss_part,
                                                    int n_part, float* __restrict__ g, float* __restrict__ loss,
                                                    const uint32_t* __restrict__ err) {
    __shared__ float4 sh[8][32];
    const bool failed = *err != 0u;   // some CTA left no partial sums: the gradient stays, the loss is NaN
    const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + c;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < kParams / 4) {
#pragma unroll 4
        for (int p = w; p < n_part; p += 8) {
            const float4 v = reinterpret_cast<const float4*>(part + (size_t)p * kParams)[i];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
    }
    sh[w][c] = a;
    __syncthreads();
    if (w == 0 && i < kParams / 4 && !failed) {
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            const float4 v = sh[q][c];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
        reinterpret_cast<float4*>(g)[i] = a;
    }
    if (loss != nullptr && blockIdx.x == 0 && w == 1) {
        double t = 0.0;
        for (int p = c; p < n_part; p += 32) t += loss_part[p];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        if (c == 0) *loss = failed ? NAN : (float)t;
    }
}

// A parameter's place(s) in the bf16 weight image (biases have none)
__device__ __forceinline__ void store_weight(uint8_t* img, int i, float v) {
    const bf16 h = __float2bfloat16_rn(v);
    auto put = [&](uint32_t off) { *reinterpret_cast<bf16*>(img + off) = h; };
    if (i < kOffB1) {
        put(kImgW1 + core_off<kIn>(i / kIn, i % kIn));
    } else if (i >= kOffW2 && i < kOffB2) {
        const int r = (i - kOffW2) / kHid, k = (i - kOffW2) % kHid;
        put(kImgW2 + core_off<kHid>(r, k));
        put(kImgW2T + core_off<kHid>(k, r));
    } else if (i >= kOffW3 && i < kOffB3) {
        const int r = (i - kOffW3) / kHid, k = (i - kOffW3) % kHid;
        put(kImgW3 + core_off<kHid>(r, k));
        put(kImgW3T + core_off<kOutPad>(k, r));
    }
}

__global__ void k_mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float bc1,
                           float bc2, uint8_t* __restrict__ img, const uint32_t* __restrict__ err) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t failed = *err;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi, vi = b2 * v[i] + (1.f - b2) * gi * gi;
    if (failed != 0u) return;   // the gradient is not that of the last backward
    m[i] = mi;
    v[i] = vi;
    const float w = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    p[i] = w;
    store_weight(img, i, w);
}

__global__ void k_weight_image(const float* __restrict__ p, uint8_t* __restrict__ img) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kParams) store_weight(img, i, p[i]);
}

// MLP input of each point: 5x5 RGB patch around its nearest pixel (clamped to the
// image; row-major, RGB interleaved), depth, camera-frame position, 0.
// One warp a point: lanes load the patch side by side (a thread that walked the 75 values alone took
// 12 us for 96 points; 4 us).
__global__ void __launch_bounds__(128) k_features(DevCamera cam, const float* __restrict__ image,
                                                  const float* __restrict__ pts, int n, float* __restrict__ f) {
    const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n) return;
    const float x = pts[3 * i], y = pts[3 * i + 1], z = pts[3 * i + 2];
    const float tx = cam.R[0] * x + cam.R[1] * y + cam.R[2] * z + cam.t[0];
    const float ty = cam.R[3] * x + cam.R[4] * y + cam.R[5] * z + cam.t[1];
    const float tz = cam.R[6] * x + cam.R[7] * y + cam.R[8] * z + cam.t[2];
    const float zz = tz > 1e-6f ? tz : 1e-6f;
    const float u = cam.fx * tx / zz + cam.cx, v = cam.fy * ty / zz + cam.cy;
    const int px = (int)fminf(fmaxf(floorf(u + 0.5f), 0.f), (float)(cam.width - 1));
    const int py = (int)fminf(fmaxf(floorf(v + 0.5f), 0.f), (float)(cam.height - 1));
    const size_t HW = (size_t)cam.width * cam.height;
    float* o = f + (size_t)i * kIn;
#pragma unroll
    for (int k = lane; k < kIn; k += 32) {
        float val;
        if (k < 75) {
            const int q = k / 3, ch = k - 3 * q, dy = q / 5 - 2, dx = q - 5 * (q / 5) - 2;
            const int xx = min(max(px + dx, 0), cam.width - 1), yy = min(max(py + dy, 0), cam.height - 1);
            val = image[(size_t)ch * HW + (size_t)yy * cam.width + xx];
        } else {
            val = k == 76 ? tx : (k == 77 ? ty : (k == 79 ? 0.f : tz));
        }
        o[k] = val;
    }
}

// Gaussian parameters [14][cap] columns base.. of the kept points from the MLP
// outputs [n][16]; a point whose prediction is non-finite or whose log-scale
// leaves [-9, 1] keeps the plain initialisation already staged for it.
__global__ void k_apply_mlp(const float* __restrict__ y, const float* __restrict__ pts, int n,
                            float* __restrict__ stage) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float* o = y + (size_t)i * kOutPad;
    bool ok = true;
    for (int c = 0; c < kOut; ++c) ok = ok && isfinite(o[c]);
    for (int c = 0; c < 3; ++c) ok = ok && o[c] >= -9.f && o[c] <= 1.f;
    const float qn = o[3] * o[3] + o[4] * o[4] + o[5] * o[5] + o[6] * o[6];
    ok = ok && qn > 1e-8f;
    if (!ok) return;
    for (int c = 0; c < 11; ++c) stage[(size_t)(3 + c) * n + i] = o[c];
}

// Training target of the learned initialiser for Gaussian `first + i` of the
// planar [14][cap] parameters: [log-scale (3), unit quaternion with w >= 0
// (q and -q are the same rotation), opacity logit, colour (3), 0 x 5]. A zero
// quaternion stays zero.
__global__ void k_mlp_targets(const float* __restrict__ P, int cap, int first, int count, float* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const size_t j = (size_t)first + i;
    const size_t C = (size_t)cap;
    float* o = out + (size_t)i * kOutPad;
    const float w = P[6 * C + j], x = P[7 * C + j], y = P[8 * C + j], z = P[9 * C + j];
    const float nrm = sqrtf(w * w + x * x + y * y + z * z);
    const float inv = nrm > 0.f ? (w < 0.f ? -1.f : 1.f) / nrm : 0.f;
    o[0] = P[3 * C + j];
    o[1] = P[4 * C + j];
    o[2] = P[5 * C + j];
    o[3] = w * inv;
    o[4] = x * inv;
    o[5] = y * inv;
    o[6] = z * inv;
    o[7] = P[10 * C + j];
    o[8] = P[11 * C + j];
    o[9] = P[12 * C + j];
    o[10] = P[13 * C + j];
#pragma unroll
    for (int k = kOut; k < kOutPad; ++k) o[k] = 0.f;
}

}  // namespace
}  // namespace gs

using namespace gs;

struct gs_mlp {
    int device = 0;
    int num_sms = 1;
    float* p = nullptr;      // f32 master parameters [kParams]
    float* g = nullptr;      // gradient
    float* m = nullptr;
    float* v = nullptr;
    uint8_t* img = nullptr;  // bf16 weights in the kernels' shared-memory layout [kImgBytes], then derr
    int t = 0;
    int rows_cap = 0;
    float* y = nullptr;      // [rows][16] predictions for an insertion
    int part_cap = 0;
    float* part = nullptr;        // [CTAs][kParams] partial gradients
    float* loss_part = nullptr;   // [CTAs]
    // flags that a kernel sets when a wait of its gave up, pinned and on the device
    uint32_t* herr = nullptr;
    uint32_t* derr = nullptr;
    uint32_t give_up = 0;     // tests: see NetErr
};

namespace gs {
// whether a wait of an earlier launch gave up (once its stream has passed it)
bool mlp_timed_out(const gs_mlp* M) { return *(volatile const uint32_t*)M->herr != 0u; }
}  // namespace gs

namespace {

int mlp_rows(gs_mlp* M, int rows) {
    if (rows <= M->rows_cap) return GS_OK;
    cudaFree(M->y);
    M->y = nullptr;
    M->rows_cap = 0;
    const size_t r = (size_t)std::max(rows, 1024);
    if (cudaMalloc(&M->y, sizeof(float) * r * kOutPad) != cudaSuccess) {
        M->y = nullptr;
        cudaGetLastError();
        return GS_ERR_OOM;
    }
    M->rows_cap = (int)r;
    return GS_OK;
}

int mlp_parts(gs_mlp* M, int ctas) {
    if (ctas <= M->part_cap) return GS_OK;
    cudaFree(M->part);
    cudaFree(M->loss_part);
    M->part = M->loss_part = nullptr;
    M->part_cap = 0;
    if (cudaMalloc(&M->part, sizeof(float) * (size_t)ctas * kParams) != cudaSuccess ||
        cudaMalloc(&M->loss_part, sizeof(float) * (size_t)ctas) != cudaSuccess) {
        cudaFree(M->part);
        M->part = M->loss_part = nullptr;
        cudaGetLastError();
        return GS_ERR_OOM;
    }
    M->part_cap = ctas;
    return GS_OK;
}

// Passes of 32 rows while the GPU has an SM for each, else of 64 (fewer, each with twice the work
// between the same products: gradients of 4,096 rows with the reduction 20 us in 128 CTAs of 32 rows,
// 28 in 64 of 64; 96 rows forward 6.2 and 8.2 us); as many CTAs as share the passes evenly.
int net_rows(const gs_mlp* M, int rows) { return (rows + 31) / 32 <= M->num_sms ? 32 : 64; }
int net_ctas(const gs_mlp* M, int rows) {
    const int per = net_rows(M, rows), passes = (rows + per - 1) / per;
    const int rounds = (passes + M->num_sms - 1) / M->num_sms;
    return (passes + rounds - 1) / rounds;
}

template <bool TRAIN, int ROWS>
void net_launch(gs_mlp* M, const float* feat, const float* tgt, int n, float* out, cudaStream_t s) {
    k_mlp_net<TRAIN, ROWS><<<net_ctas(M, n), kNetThreads, Smem<TRAIN, ROWS>::Bytes, s>>>(
        feat, tgt, n, M->img, M->p, out, M->part, M->loss_part, NetErr{M->derr, M->herr, M->give_up});
}

template <bool TRAIN, int ROWS>
bool net_smem() {
    return cudaFuncSetAttribute(k_mlp_net<TRAIN, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                Smem<TRAIN, ROWS>::Bytes) == cudaSuccess;
}

// predictions out [rows][16] of feature rows (f32 [rows][80])
cudaError_t mlp_forward_rows(gs_mlp* M, const float* feat, int rows, float* out, cudaStream_t s) {
    if (net_rows(M, rows) == 32) net_launch<false, 32>(M, feat, nullptr, rows, out, s);
    else net_launch<false, 64>(M, feat, nullptr, rows, out, s);
    return cudaGetLastError();
}

}  // namespace

// ---------------------------------------------------------------- C ABI

extern "C" {

int gs_mlp_targets(gs_ctx* c, int first, int count, float* out_dev, void* stream) {
    if (!c || first < 0 || count < 0 || first > c->n || count > c->n - first || (count > 0 && !out_dev))
        return GS_ERR_ARG;
    if (count == 0) return GS_OK;
    if (cudaSetDevice(c->device) != cudaSuccess) return GS_ERR_CUDA;
    ++c->launches;
    k_mlp_targets<<<(count + 255) / 256, 256, 0, (cudaStream_t)stream>>>(c->params, c->cap, first, count, out_dev);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

int gs_mlp_create(int device, uint64_t seed, gs_mlp** out) {
    if (!out) return GS_ERR_ARG;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return GS_ERR_CUDA;
    gs_mlp* M = new gs_mlp();
    M->device = device;
    bool ok = cudaMalloc(&M->p, sizeof(float) * kParams) == cudaSuccess;
    ok = ok && cudaMalloc(&M->g, sizeof(float) * kParams) == cudaSuccess;
    ok = ok && cudaMalloc(&M->m, sizeof(float) * kParams) == cudaSuccess;
    ok = ok && cudaMalloc(&M->v, sizeof(float) * kParams) == cudaSuccess;
    ok = ok && cudaMalloc(&M->img, kImgBytes + sizeof(uint32_t)) == cudaSuccess;
    if (ok) M->derr = reinterpret_cast<uint32_t*>(M->img + kImgBytes);
    ok = ok && cudaMemset(M->derr, 0, sizeof(uint32_t)) == cudaSuccess;
    ok = ok && cudaMallocHost((void**)&M->herr, sizeof(uint32_t)) == cudaSuccess;
    if (ok) *M->herr = 0u;
    if (!ok) {
        gs_mlp_destroy(M);
        return GS_ERR_OOM;
    }
    if (cudaDeviceGetAttribute(&M->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || M->num_sms < 1)
        M->num_sms = 1;
    if (!net_smem<false, 32>() || !net_smem<false, 64>() || !net_smem<true, 32>() || !net_smem<true, 64>()) {
        cudaGetLastError();
        gs_mlp_destroy(M);
        return GS_ERR_CUDA;
    }
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights from SplitMix64, zero biases; output rows >= 11 zero
    float* h = (float*)calloc(kParams, sizeof(float));
    uint64_t st = seed;
    auto uni = [&st]() {
        st += 0x9E3779B97F4A7C15ull;
        uint64_t z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    for (int i = 0; i < kHid * kIn; ++i) h[kOffW1 + i] = (float)((2 * uni() - 1) / std::sqrt((double)kIn));
    for (int i = 0; i < kHid * kHid; ++i) h[kOffW2 + i] = (float)((2 * uni() - 1) / std::sqrt((double)kHid));
    for (int i = 0; i < kOut * kHid; ++i) h[kOffW3 + i] = (float)((2 * uni() - 1) / std::sqrt((double)kHid));
    cudaError_t e = cudaMemcpy(M->p, h, sizeof(float) * kParams, cudaMemcpyHostToDevice);
    free(h);
    if (e == cudaSuccess) e = gs_mlp_set_params(M, M->p, nullptr) == GS_OK ? cudaSuccess : cudaErrorUnknown;
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        gs_mlp_destroy(M);
        return GS_ERR_CUDA;
    }
    *out = M;
    return GS_OK;
}

void gs_mlp_destroy(gs_mlp* M) {
    if (!M) return;
    cudaSetDevice(M->device);
    void* ps[] = {M->p, M->g, M->m, M->v, M->img, M->y, M->part, M->loss_part};
    for (void* q : ps) cudaFree(q);
    if (M->herr) cudaFreeHost(M->herr);
    delete M;
}

int gs_mlp_set_params(gs_mlp* M, const float* flat_dev, void* stream) {
    if (!M || !flat_dev) return GS_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (flat_dev != M->p && cudaMemcpyAsync(M->p, flat_dev, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, s) !=
                                cudaSuccess)
        return GS_ERR_CUDA;
    cudaMemsetAsync(M->m, 0, sizeof(float) * kParams, s);
    cudaMemsetAsync(M->v, 0, sizeof(float) * kParams, s);
    cudaMemsetAsync(M->g, 0, sizeof(float) * kParams, s);
    M->t = 0;
    k_weight_image<<<(kParams + 255) / 256, 256, 0, s>>>(M->p, M->img);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

int gs_mlp_get_params(gs_mlp* M, float* flat_dev, void* stream) {
    if (!M || !flat_dev) return GS_ERR_ARG;
    return cudaMemcpyAsync(flat_dev, M->p, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, (cudaStream_t)stream) ==
                   cudaSuccess
               ? GS_OK
               : GS_ERR_CUDA;
}

int gs_mlp_get_grads(gs_mlp* M, float* flat_dev, void* stream) {
    if (!M || !flat_dev) return GS_ERR_ARG;
    return cudaMemcpyAsync(flat_dev, M->g, sizeof(float) * kParams, cudaMemcpyDeviceToDevice, (cudaStream_t)stream) ==
                   cudaSuccess
               ? GS_OK
               : GS_ERR_CUDA;
}

int gs_mlp_features(const gs_camera* cam, const float* image_dev, const float* points_dev, int n, float* feat_dev,
                    void* stream) {
    if (n < 0 || (n > 0 && (!cam || !image_dev || !points_dev || !feat_dev))) return GS_ERR_ARG;
    if (n == 0) return GS_OK;
    if (cam->width <= 0 || cam->height <= 0) return GS_ERR_ARG;
    DevCamera d;
    memset(&d, 0, sizeof(d));
    memcpy(d.R, cam->R, sizeof(d.R));
    memcpy(d.t, cam->t, sizeof(d.t));
    d.fx = cam->fx;
    d.fy = cam->fy;
    d.cx = cam->cx;
    d.cy = cam->cy;
    d.width = cam->width;
    d.height = cam->height;
    k_features<<<(n + 3) / 4, 128, 0, (cudaStream_t)stream>>>(d, image_dev, points_dev, n, feat_dev);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

int gs_mlp_forward(gs_mlp* M, const float* feat_dev, int n, float* out_dev, void* stream) {
    if (!M || n < 0 || (n > 0 && (!feat_dev || !out_dev))) return GS_ERR_ARG;
    if (n == 0) return GS_OK;
    if (mlp_timed_out(M)) return GS_ERR_TIMEOUT;   // a wait of an earlier call gave up
    return mlp_forward_rows(M, feat_dev, n, out_dev, (cudaStream_t)stream) == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

int gs_mlp_backward(gs_mlp* M, const float* feat_dev, const float* target_dev, int n, float* loss_dev, void* stream) {
    if (!M || n <= 0 || !feat_dev || !target_dev) return GS_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (mlp_timed_out(M)) return GS_ERR_TIMEOUT;   // a wait of an earlier call gave up
    const int ctas = net_ctas(M, n);
    if (mlp_parts(M, ctas) != GS_OK) return GS_ERR_OOM;
    if (net_rows(M, n) == 32) net_launch<true, 32>(M, feat_dev, target_dev, n, nullptr, s);
    else net_launch<true, 64>(M, feat_dev, target_dev, n, nullptr, s);
    k_mlp_reduce<<<(kParams / 4 + 31) / 32, 256, 0, s>>>(M->part, M->loss_part, ctas, M->g, loss_dev,
                                                             M->derr);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

int gs_mlp_step(gs_mlp* M, float lr, void* stream) {
    if (!M || !(lr > 0.f)) return GS_ERR_ARG;
    if (mlp_timed_out(M)) return GS_ERR_TIMEOUT;
    cudaStream_t s = (cudaStream_t)stream;
    M->t += 1;
    const double b1 = 0.9, b2 = 0.999;
    k_mlp_adam<<<(kParams + 255) / 256, 256, 0, s>>>(M->p, M->g, M->m, M->v, kParams, lr, (float)b1, (float)b2, 1e-8f,
                                                     (float)(1.0 - std::pow(b1, M->t)), (float)(1.0 - std::pow(b2, M->t)),
                                                     M->img, M->derr);
    return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

int gs_mlp_num_params(void) { return kParams; }

int gs_debug_mlp_give_up(gs_mlp* M, int nth) {
    if (!M || nth < 0) return GS_ERR_ARG;
    M->give_up = (uint32_t)nth;
    return GS_OK;
}

}  // extern "C"

namespace gs {

// Learned initial parameters for the staged points [14][n] (plain values stay where the MLP
// gives none): features -> MLP -> k_apply_mlp.
cudaError_t mlp_initialise(gs_mlp* M, const DevCamera& cam, const float* image, const float* pts, int n, float* stage,
                           float* feat_tmp, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if (mlp_rows(M, n) != GS_OK) return cudaErrorMemoryAllocation;
    k_features<<<(n + 3) / 4, 128, 0, s>>>(cam, image, pts, n, feat_tmp);
    cudaError_t e = mlp_forward_rows(M, feat_tmp, n, M->y, s);
    if (e != cudaSuccess) return e;
    k_apply_mlp<<<(n + 127) / 128, 128, 0, s>>>(M->y, pts, n, stage);
    return cudaGetLastError();
}

}  // namespace gs
