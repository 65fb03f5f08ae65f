// Tile binning and the (tile, depth) ordering of the pairs.
//
// The order the compositing needs is lexicographic in (view, tile, depth,
// Gaussian id). It is built in two stable steps instead of one 64-bit sort:
//   1. a stable LSD radix sort of the visible items' depth keys, three passes
//      over the bits their range needs (nine bits a pass for depths up to 2^16
//      times the nearest, at most eleven), whose stability keeps equal depths
//      in id order; maps of at most kSmallItems (view, Gaussian) items do it in
//      one CTA;
//   2. pairs are emitted in that depth order (one per tile a Gaussian's pixel
//      box touches), then stably radix-sorted by bin = view * tiles + tile
//      (2 passes for up to 65536 bins).
// The second sort moves 8-byte pairs over P elements only twice instead of six
// times for a 64-bit key, and the depth sort touches N elements, not P.
//
// Every pass is reduce-then-scan over a fixed grid of G blocks, each owning a
// contiguous slice of the input: one launch counts digits per block, the next
// adds the counts it needs itself (of many blocks, a launch between them does)
// and scatters. Element counts (and the depth
// keys' range) are read from device memory so the same launches can sit in a
// CUDA graph. These launches move a few MB at most; what they cost is the
// launches and their dependent latencies.
#include <algorithm>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 8;                       // per lane per round
constexpr int kRound = kSortThreads * kSortItems;   // elements per block round

__device__ __forceinline__ void slice_of(uint32_t n, int G, int b, uint32_t& begin, uint32_t& end) {
    uint32_t chunk = (n + G - 1) / G;
    chunk = (chunk + 31u) & ~31u;
    uint64_t b0 = (uint64_t)chunk * b, b1 = b0 + chunk;
    begin = (uint32_t)(uint32_t)(b0 < n ? b0 : n);
    end = (uint32_t)(uint32_t)(b1 < n ? b1 : n);
}

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The digit of one pass: the low `bits` bits of key - base in `passes` passes of equal width, with
// bits given, or base and bits from the keys' {min, max} on the device.
struct DigitSpec {
    const uint32_t* range;
    int bits, pass, passes;
};
struct Digit {
    uint32_t base, mask;
    int shift, nbits;
    __device__ __forceinline__ Digit(const DigitSpec& s) {
        base = 0;
        int bits = s.bits;
        if (s.range != nullptr) {
            base = s.range[0];
            bits = 32 - __clz(s.range[1] - base);
        }
        const int w = (bits + s.passes - 1) / s.passes;
        shift = s.pass * w;
        nbits = max(min(w, bits - shift), 0);
        if (nbits == 0) shift = 0;
        mask = (1u << nbits) - 1u;
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t key) const { return ((key - base) >> shift) & mask; }
};

// Histogram of one digit over each block's slice: hist[b << nbits | d]. Up to eight shared
// sub-histograms, one a warp (shared-memory atomics); every thread has four keys in flight.
template <int MAXBITS>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint32_t* __restrict__ keys,
                                                             const uint32_t* __restrict__ n_dev, uint32_t n_max,
                                                             DigitSpec spec, uint32_t* __restrict__ hist) {
    constexpr int kWords = kSortWarps << (MAXBITS <= 8 ? MAXBITS : 9);
    __shared__ uint32_t h[kWords];
    const int G = gridDim.x, b = blockIdx.x;
    uint32_t n = umin(*n_dev, n_max), begin, end;
    slice_of(n, G, b, begin, end);
    const Digit dig(spec);
    const int nsub = min(kSortWarps, kWords >> dig.nbits);
    for (int d = threadIdx.x; d < nsub << dig.nbits; d += kSortThreads) h[d] = 0;
    __syncthreads();
    uint32_t* hw = h + (((threadIdx.x >> 5) & (nsub - 1)) << dig.nbits);
    for (uint32_t base = begin + threadIdx.x; base < end; base += 4 * kSortThreads) {
        uint32_t k[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t i = base + u * kSortThreads;
            k[u] = i < end ? keys[i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (base + u * kSortThreads < end) atomicAdd(&hw[dig(k[u])], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d <= (int)dig.mask; d += kSortThreads) {
        uint32_t t = 0;
        for (int q = 0; q < nsub; ++q) t += h[(q << dig.nbits) + d];
        hist[((size_t)b << dig.nbits) + d] = t;
    }
}

// Of more than kScanGrid blocks (at most kMaxGrid): the rows' exclusive scan over the blocks, in place,
// and each digit's total. A CTA takes eight digits, 32 threads each; a thread's rows are loaded
// together and stay in registers.
constexpr int kScanGrid = 128, kScanRows = 20, kMaxGrid = 32 * kScanRows;
__global__ void __launch_bounds__(256) k_digit_scan(uint32_t* __restrict__ hist, int G, DigitSpec spec,
                                                    uint32_t* __restrict__ dtot) {
    __shared__ uint32_t part[32][8];
    const Digit dig(spec);
    const int c = threadIdx.x & 7, g = threadIdx.x >> 3;
    const int d = blockIdx.x * 8 + c, ndig = 1 << dig.nbits;
    if (blockIdx.x * 8 >= ndig) return;   // the whole CTA (the grid is for the widest digit)
    const int chunk = (G + 31) / 32, r0 = g * chunk, rows = d < ndig ? min(chunk, G - r0) : 0;
    uint32_t* col = hist + ((size_t)r0 << dig.nbits) + d;
    uint32_t v[kScanRows], sum = 0;
#pragma unroll
    for (int r = 0; r < kScanRows; ++r) v[r] = r < rows ? col[(size_t)r << dig.nbits] : 0u;
#pragma unroll
    for (int r = 0; r < kScanRows; ++r) sum += v[r];
    part[g][c] = sum;
    __syncthreads();
    uint32_t run = 0, all = 0;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
        const uint32_t x = part[q][c];
        run += q < g ? x : 0u;
        all += x;
    }
#pragma unroll
    for (int r = 0; r < kScanRows; ++r) {
        if (r < rows) col[(size_t)r << dig.nbits] = run;
        run += v[r];
    }
    if (g == 0 && d < ndig) dtot[d] = all;
}

// Stable scatter of one digit pass. Up to kScanGrid blocks the block first adds the digit counts of
// the blocks before its own, and of all blocks, straight from the histogram rows (16-byte loads, rows
// in parallel: less than a separate scan launch takes; at 608 blocks and 128 digits it took 25 us more
// than the scan), else it finds them in its row and in dtot. Then it
// walks its slice in rounds of kRound elements; warp w of a round owns a contiguous run of
// 32*kSortItems elements, ranked within the warp by __match_any_sync, across warps by a
// per-digit prefix over the warps' counts, and across blocks by those sums.
// The ranked round is first regrouped by digit in shared memory,
// then written out by consecutive threads, so each digit's run of the round
// leaves in coalesced stores instead of one scattered store per element.
template <int MAXBITS>
struct ScatterSmem {
    static constexpr int D = 1 << MAXBITS;
    uint32_t run[D];      // global position of the block's next element of each digit
    uint32_t lstart[D];   // start of each digit's group in the staged round
    uint16_t wcnt[kSortWarps][D];
    uint32_t skey[kRound], sval[kRound];
    uint32_t wsum[kSortWarps];
};
template <int MAXBITS>
__global__ void __launch_bounds__(kSortThreads, MAXBITS <= 8 ? 5 : 3) k_radix_scatter(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, const uint32_t* __restrict__ n_dev, uint32_t n_max, DigitSpec spec,
    const uint32_t* __restrict__ hist, const uint32_t* __restrict__ dtot) {
    extern __shared__ __align__(16) uint8_t scatter_smem[];
    ScatterSmem<MAXBITS>& sm = *reinterpret_cast<ScatterSmem<MAXBITS>*>(scatter_smem);
    constexpr int E = (1 << MAXBITS) / kSortThreads < 1 ? 1 : (1 << MAXBITS) / kSortThreads;   // digits a thread
    const int G = gridDim.x, b = blockIdx.x, t = threadIdx.x;
    const Digit dig(spec);
    const int ndig = 1 << dig.nbits;
    const int lane = t & 31, w = t >> 5;
    // exclusive scan of one value per thread over the block
    auto block_scan = [&](uint32_t c) -> uint32_t {
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sm.wsum[w] = x;
        __syncthreads();
        uint32_t pre = 0;
        for (int k = 0; k < w; ++k) pre += sm.wsum[k];
        __syncthreads();
        return pre + x - c;
    };
    // run: counts before this block; lstart: totals
    for (int d = t; d < ndig; d += kSortThreads) {
        sm.run[d] = dtot != nullptr ? hist[((size_t)b << dig.nbits) + d] : 0u;
        sm.lstart[d] = dtot != nullptr ? dtot[d] : 0u;
    }
    __syncthreads();
    if (dtot != nullptr) {
    } else if (dig.nbits >= 2) {
        const int cols = ndig / 4, groups = max(1, kSortThreads / cols);
        for (int c = t % min(cols, kSortThreads); c < cols; c += kSortThreads) {
            uint4 bef = make_uint4(0, 0, 0, 0), tot = bef;
            const uint4* row = reinterpret_cast<const uint4*>(hist) + c;
            constexpr int R = MAXBITS <= 8 ? 8 : 16;   // rows in flight
            for (int r0 = t / min(cols, kSortThreads); r0 < G; r0 += R * groups) {
                uint4 v[R];
#pragma unroll
                for (int u = 0; u < R; ++u) {
                    const int r = r0 + u * groups;
                    v[u] = r < G ? row[(size_t)r * cols] : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int u = 0; u < R; ++u) {
                    const bool before = r0 + u * groups < b;
                    tot.x += v[u].x;
                    tot.y += v[u].y;
                    tot.z += v[u].z;
                    tot.w += v[u].w;
                    bef.x += before ? v[u].x : 0u;
                    bef.y += before ? v[u].y : 0u;
                    bef.z += before ? v[u].z : 0u;
                    bef.w += before ? v[u].w : 0u;
                }
            }
            const uint32_t vb[4] = {bef.x, bef.y, bef.z, bef.w}, vt[4] = {tot.x, tot.y, tot.z, tot.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                atomicAdd(&sm.run[4 * c + q], vb[q]);
                atomicAdd(&sm.lstart[4 * c + q], vt[q]);
            }
        }
    } else {
        for (int r = t; r < G; r += kSortThreads)
            for (int d = 0; d < ndig; ++d) {
                const uint32_t v = hist[(size_t)r * ndig + d];
                atomicAdd(&sm.lstart[d], v);
                if (r < b) atomicAdd(&sm.run[d], v);
            }
    }
    __syncthreads();
    {   // thread t holds digits t * per .. : exclusive scan of the totals
        const int per = max(1, ndig / kSortThreads);
        uint32_t v[E], sum = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int d = t * per + e;
            v[e] = e < per && d < ndig ? sm.lstart[d] : 0u;
            sum += v[e];
        }
        uint32_t start = block_scan(sum);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int d = t * per + e;
            if (e < per && d < ndig) sm.run[d] += start;
            start += v[e];
        }
    }
    __syncthreads();
    uint32_t n = umin(*n_dev, n_max), begin, end;
    slice_of(n, G, b, begin, end);
    const uint32_t lt = lanemask_lt();
    for (uint32_t rbase = begin; rbase < end; rbase += kRound) {
        for (int d = lane; d < ndig; d += 32) sm.wcnt[w][d] = 0;
        __syncwarp();
        uint32_t key[kSortItems], val[kSortItems], rank[kSortItems];
        const uint32_t wbase = rbase + (uint32_t)w * 32u * kSortItems;
#pragma unroll
        for (int it = 0; it < kSortItems; ++it) {
            uint32_t i = wbase + it * 32 + lane;
            bool ok = i < end;
            key[it] = ok ? kin[i] : 0u;
            val[it] = ok ? vin[i] : 0u;
        }
#pragma unroll
        for (int it = 0; it < kSortItems; ++it) {
            const bool ok = wbase + it * 32 + lane < end;
            uint32_t d = ok ? dig(key[it]) : 0xFFFFFFFFu;
            uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
            uint32_t r = 0;
            if (ok) r = sm.wcnt[w][d] + __popc(peers & lt);
            rank[it] = r;
            __syncwarp();
            if (ok && (__ffs(peers) - 1) == lane) sm.wcnt[w][d] += (uint16_t)__popc(peers);
            __syncwarp();
        }
        __syncthreads();
        // per digit: prefix over the warps, the round's count, and its group start in the round
        uint32_t tot[E];
        {
            const int per = max(1, ndig / kSortThreads);
            uint32_t sum = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int d = t * per + e;
                tot[e] = 0;
                if (e < per && d < ndig) {
#pragma unroll
                    for (int ww = 0; ww < kSortWarps; ++ww) {
                        const uint32_t c = sm.wcnt[ww][d];
                        sm.wcnt[ww][d] = (uint16_t)tot[e];
                        tot[e] += c;
                    }
                }
                sum += tot[e];
            }
            uint32_t ls = block_scan(sum);   // synchronises the block
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int d = t * per + e;
                if (e < per && d < ndig) sm.lstart[d] = ls;
                ls += tot[e];
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kSortItems; ++it) {
            const uint32_t i = wbase + it * 32 + lane;
            if (i < end) {
                const uint32_t d = dig(key[it]);
                const uint32_t lp = sm.lstart[d] + sm.wcnt[w][d] + rank[it];
                sm.skey[lp] = key[it];
                sm.sval[lp] = val[it];
            }
        }
        __syncthreads();
        const uint32_t cnt = umin((uint32_t)kRound, end - rbase);
        for (uint32_t j = t; j < cnt; j += kSortThreads) {
            const uint32_t k2 = sm.skey[j], d = dig(k2);
            const uint32_t pos = sm.run[d] + (j - sm.lstart[d]);
            kout[pos] = k2;
            vout[pos] = sm.sval[j];
        }
        __syncthreads();
        {
            const int per = max(1, ndig / kSortThreads);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int d = t * per + e;
                if (e < per && d < ndig) sm.run[d] += tot[e];
            }
        }
        __syncthreads();
    }
}

template <int MAXBITS>
cudaError_t launch_radix_pass(int G, const uint32_t* kin, const uint32_t* vin, uint32_t* kout, uint32_t* vout,
                              const uint32_t* n_dev, uint32_t n_max, const DigitSpec& spec, uint32_t* hist,
                              uint32_t* dtot, cudaStream_t s) {
    k_radix_hist<MAXBITS><<<G, kSortThreads, 0, s>>>(kin, n_dev, n_max, spec, hist);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (G > kScanGrid) {
        k_digit_scan<<<(1 << MAXBITS) / 8, 256, 0, s>>>(hist, G, spec, dtot);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    } else {
        dtot = nullptr;
    }
    k_radix_scatter<MAXBITS><<<G, kSortThreads, sizeof(ScatterSmem<MAXBITS>), s>>>(kin, vin, kout, vout, n_dev, n_max,
                                                                                  spec, hist, dtot);
    return cudaGetLastError();
}

// ---- small maps: the visible items compacted and depth-sorted in one CTA ----
//
// Raw keys and items 0 .. n - 1 in, the order and the tile counts' sums per 256 ordered items out
// (with the visible count and the pair total). In place of eight launches (compaction, three passes
// of two, tile sums) of about 3 us each.
constexpr int kSmallThreads = 1024, kSmallPer = 8, kSmallItems = kSmallThreads * kSmallPer, kSmallBits = 7;
struct SmallSmem {
    uint32_t key[kSmallItems], val[kSmallItems];
    uint16_t wcnt[32][1 << kSmallBits];
    uint32_t start[1 << kSmallBits];
    uint32_t wsum[32], kmin, kmax;
};
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_depth(const uint32_t* __restrict__ kin, uint32_t n,
                                                                 const uint32_t* __restrict__ tiles,
                                                                 uint32_t* __restrict__ order,
                                                                 uint32_t* __restrict__ tile_blocks,
                                                                 uint32_t* __restrict__ counts) {
    extern __shared__ __align__(16) uint8_t scatter_smem[];
    SmallSmem& sm = *reinterpret_cast<SmallSmem*>(scatter_smem);
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint32_t lt = lanemask_lt();
    if (t == 0) {
        sm.kmin = 0xFFFFFFFFu;
        sm.kmax = 0u;
    }
    // exclusive scan over the block of one value a warp's lane 0 (returned to the warp), and the total
    auto warps_scan = [&](uint32_t c, uint32_t& total) -> uint32_t {
        if (lane == 0) sm.wsum[w] = c;
        __syncthreads();
        const uint32_t v = sm.wsum[lane];
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        total = __shfl_sync(0xFFFFFFFFu, x, 31);
        const uint32_t e = __shfl_sync(0xFFFFFFFFu, x - v, w);
        __syncthreads();
        return e;
    };
    uint32_t key[kSmallPer], val[kSmallPer], rank[kSmallPer];
    uint32_t m;
    {
        const int per = (int)((n + kSmallThreads - 1) / kSmallThreads);
        uint32_t bal[kSmallPer], cnt = 0, lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
        for (int it = 0; it < kSmallPer; ++it) {
            const uint32_t i = (uint32_t)(w * per + it) * 32u + lane;
            const bool in = it < per && i < n;
            key[it] = in ? kin[i] : 0xFFFFFFFFu;
            const bool vis = key[it] != 0xFFFFFFFFu;
            bal[it] = __ballot_sync(0xFFFFFFFFu, vis);
            cnt += __popc(bal[it]);
            lo = umin(lo, key[it]);
            if (vis) hi = umax(hi, key[it]);
        }
        lo = __reduce_min_sync(0xFFFFFFFFu, lo);
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);
        uint32_t pos = warps_scan(cnt, m);
        if (lane == 0) {
            atomicMin(&sm.kmin, lo);
            atomicMax(&sm.kmax, hi);
        }
#pragma unroll
        for (int it = 0; it < kSmallPer; ++it) {
            if (bal[it] >> lane & 1u) {
                const uint32_t p = pos + __popc(bal[it] & lt);
                sm.key[p] = key[it];
                sm.val[p] = (uint32_t)(w * per + it) * 32u + lane;
            }
            pos += __popc(bal[it]);
        }
    }
    __syncthreads();
    const uint32_t base = sm.kmin;
    const int bits = m ? 32 - __clz(sm.kmax - base) : 0;
    const int passes = (bits + kSmallBits - 1) / kSmallBits, width = passes ? (bits + passes - 1) / passes : 0;
    const int ndig = 1 << width;
    const uint32_t mask = (uint32_t)ndig - 1u;
    const int per = (int)((m + kSmallThreads - 1) / kSmallThreads);
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * width;
        for (int d = lane; d < ndig; d += 32) sm.wcnt[w][d] = 0;
        __syncwarp();
#pragma unroll
        for (int it = 0; it < kSmallPer; ++it) {
            if (it >= per) break;
            const uint32_t i = (uint32_t)(w * per + it) * 32u + lane;
            const bool ok = i < m;
            key[it] = ok ? sm.key[i] : 0u;
            val[it] = ok ? sm.val[i] : 0u;
            const uint32_t d = ok ? ((key[it] - base) >> shift) & mask : 0xFFFFFFFFu;
            const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
            rank[it] = ok ? sm.wcnt[w][d] + __popc(peers & lt) : 0u;
            __syncwarp();
            if (ok && (__ffs(peers) - 1) == lane) sm.wcnt[w][d] += (uint16_t)__popc(peers);
            __syncwarp();
        }
        __syncthreads();
        uint32_t tot = 0;
        if (t < ndig) {
#pragma unroll 8
            for (int ww = 0; ww < 32; ++ww) {
                const uint32_t c = sm.wcnt[ww][t];
                sm.wcnt[ww][t] = (uint16_t)tot;
                tot += c;
            }
        }
        uint32_t x = tot;   // digits 32 w + lane: inclusive scan in the warp, then over the warps
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        uint32_t all;
        const uint32_t pre = warps_scan(__shfl_sync(0xFFFFFFFFu, x, 31), all);
        if (t < ndig) sm.start[t] = pre + x - tot;
        __syncthreads();
#pragma unroll
        for (int it = 0; it < kSmallPer; ++it) {
            if (it >= per) break;
            const uint32_t i = (uint32_t)(w * per + it) * 32u + lane;
            if (i < m) {
                const uint32_t d = ((key[it] - base) >> shift) & mask;
                const uint32_t p = sm.start[d] + sm.wcnt[w][d] + rank[it];
                sm.key[p] = key[it];
                sm.val[p] = val[it];
            }
        }
        __syncthreads();
    }
    unsigned long long total = 0;   // (threads 0 .. 3: their blocks')
    // tile counts per 256 ordered items (eight warps of 32 a block): sums for the emission
    for (uint32_t i0 = 0; i0 < m; i0 += kSmallThreads) {
        const uint32_t i = i0 + t;
        uint32_t c = 0;
        if (i < m) {
            const uint32_t item = sm.val[i];
            order[i] = item;
            c = tiles[item];
        }
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (lane == 0) sm.wsum[w] = c;
        __syncthreads();
        if (t < 4 && i0 + 256u * t < m) {
            unsigned long long b = 0;
            for (int q = 0; q < 8; ++q) b += sm.wsum[8 * t + q];
            tile_blocks[i0 / 256 + t] = (uint32_t)b;
            total += b;
        }
        __syncthreads();
    }
    if (t < 4) {
        total += __shfl_xor_sync(0xFu, total, 1);
        total += __shfl_xor_sync(0xFu, total, 2);
    }
    if (t == 0) {
        counts[0] = (uint32_t)total;
        counts[1] = (uint32_t)(total >> 32);
        counts[8] = m;
    }
}

// Tiles touched by each 256 items of the depth order (the emission's CTAs), and their total in 64 bits
// (a map that fills the screen can have more than 2^32 pairs; nothing is emitted then).
__global__ void __launch_bounds__(256) k_item_tiles(const uint32_t* __restrict__ order,
                                                    const uint32_t* __restrict__ tiles, uint32_t n_items,
                                                    const uint32_t* __restrict__ n_dev,
                                                    uint32_t* __restrict__ tile_blocks,
                                                    unsigned long long* __restrict__ total) {
    __shared__ uint32_t ws[8];
    const uint32_t nv = umin(n_items, *n_dev);
    for (uint32_t b = blockIdx.x; b * 256u < nv; b += gridDim.x) {
        const uint32_t k = b * 256u + threadIdx.x;
        const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, k < nv ? tiles[order[k]] : 0u);
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long t = 0;
            for (int q = 0; q < 8; ++q) t += ws[q];
            tile_blocks[b] = (uint32_t)t;
            atomicAdd(total, t);   // (zeroed by the compaction)
        }
        __syncthreads();
    }
}

// ---- exclusive scan of u32 values (map management, and the tile counts of large maps) ----

__global__ void __launch_bounds__(256) k_block_sums(const uint32_t* __restrict__ in, uint32_t n,
                                                    uint32_t* __restrict__ bsum) {
    __shared__ uint32_t ws[8];
    uint32_t begin, end;
    slice_of(n, gridDim.x, blockIdx.x, begin, end);
    uint32_t s = 0;
    for (uint32_t i = begin + threadIdx.x; i < end; i += 256) s += in[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int k = 0; k < 8; ++k) t += ws[k];
        bsum[blockIdx.x] = t;
    }
}

// Exclusive scan of the slices of k_block_sums: block b first adds the block sums of the
// slices before its own (a few hundred values, read straight from bsum: no separate scan
// launch), then scans its slice; the last block writes the total.
__global__ void __launch_bounds__(256) k_scan(const uint32_t* __restrict__ in, uint32_t n,
                                              const uint32_t* __restrict__ bsum, uint32_t* __restrict__ off,
                                              uint32_t* __restrict__ total_out) {
    __shared__ uint32_t ws[8];
    __shared__ uint32_t carry;
    uint32_t begin, end;
    slice_of(n, gridDim.x, blockIdx.x, begin, end);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    {
        uint32_t pre = 0;
        for (int b = threadIdx.x; b < (int)blockIdx.x; b += 256) pre += bsum[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pre += __shfl_xor_sync(0xFFFFFFFFu, pre, o);
        if (lane == 0) ws[w] = pre;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t t = 0;
            for (int k = 0; k < 8; ++k) t += ws[k];
            carry = t;
        }
        __syncthreads();
    }
    for (uint32_t base = begin; base < end; base += 256) {
        uint32_t i = base + threadIdx.x;
        uint32_t c = i < end ? in[i] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[w] = x;
        __syncthreads();
        uint32_t pre = 0, tot = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            uint32_t v = ws[k];
            pre += (k < w) ? v : 0u;
            tot += v;
        }
        if (i < end) off[i] = carry + pre + x - c;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (total_out != nullptr && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total_out = carry;
}

// Pair emission: item k of the depth order owns pairs o .. o + tiles - 1, with o
// the tiles of the items before it (the CTA adds the block sums before its own,
// or reads their scan where `scanned`, and scans its 256 items), one per tile of
// its pixel box in row-major order (bin, item). Each warp
// takes 32 consecutive items, scans their tile counts, and writes the warp's
// pairs (a contiguous run of the output) 32 at a time: lane j writes pair t =
// t0 + j of the run, owned by the last lane whose exclusive count is <= t, so
// the stores are coalesced and a large Gaussian's pairs are spread over the
// warp. An item whose pairs would pass pair_cap is skipped and sets *overflow;
// of more than 2^32 pairs (*total_hi) every item is, since o wraps.
// In the deterministic mode (emit_item != NULL) a pair's value is its emission
// index e instead of its item, emit_item[e] holds the item, and the pair's
// gradient slot pairgrad[9 e ..] is cleared; off[k] = o for its reduction.
__global__ void __launch_bounds__(256) k_emit(const uint32_t* __restrict__ order, const uint32_t* __restrict__ tiles,
                                              const uint32_t* __restrict__ tile_blocks, bool scanned,
                                              uint32_t* __restrict__ off, const float4* __restrict__ rec,
                                              const DevCamera* __restrict__ cams, int n, int tile, uint32_t n_items,
                                              const uint32_t* __restrict__ n_dev, uint64_t pair_cap,
                                              uint32_t* __restrict__ pkey, uint32_t* __restrict__ pval,
                                              const uint32_t* __restrict__ total_hi, uint32_t* __restrict__ overflow,
                                              uint32_t* __restrict__ emit_item,
                                              float* __restrict__ pairgrad) {
    __shared__ uint32_t sbef[8], stot[8];
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t nv = umin(n_items, *n_dev);
    const bool too_many = *total_hi != 0u;
    if (blockIdx.x * blockDim.x >= nv) return;   // the whole CTA is past the visible items
    uint32_t item = 0, cnt = 0, o = 0, bin0 = 0, tiles_x = 0;
    int tx0 = 0, ty0 = 0, wt = 1;
    if (k < nv) {
        item = order[k];
        cnt = tiles[item];
    }
    {
        uint32_t bef = 0;
        if (scanned)
            bef = threadIdx.x == 0 ? tile_blocks[blockIdx.x] : 0u;
        else
            for (uint32_t b = threadIdx.x; b < blockIdx.x; b += 256) bef += tile_blocks[b];
        bef = __reduce_add_sync(0xFFFFFFFFu, bef);
        uint32_t x = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) {
            sbef[w] = bef;
            stot[w] = x;
        }
        __syncthreads();
        o = x - cnt;
#pragma unroll
        for (int q = 0; q < 8; ++q) o += sbef[q] + (q < w ? stot[q] : 0u);
    }
    if (k < nv) {
        if (emit_item != nullptr) off[k] = o;
        if (cnt != 0) {
            if (too_many || (uint64_t)o + cnt > pair_cap) {
                atomicMax(overflow, 1u);
                cnt = 0;
            } else {
                const DevCamera& cam = cams[item / (uint32_t)n];
                const float4 f0 = rec[(size_t)item * 3], f1 = rec[(size_t)item * 3 + 1],
                             f2 = rec[(size_t)item * 3 + 2];
                int x0 = 0, x1 = -1, y0 = 0, y1 = -1;
                pixel_box(f0.x, f1.w, f0.y, f2.w, f0.z, cam.width, cam.height, x0, x1, y0, y1);
                tx0 = x0 / tile;
                ty0 = y0 / tile;
                wt = x1 / tile - tx0 + 1;
                bin0 = (uint32_t)cam.bin_base;
                tiles_x = (uint32_t)cam.tiles_x;
            }
        }
    }
    uint32_t incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += y;
    }
    const uint32_t excl = incl - cnt;
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    for (uint32_t t0 = 0; t0 < total; t0 += 32) {
        const uint32_t t = t0 + (uint32_t)lane;
        int src = 0;   // last lane with excl <= t (lanes without pairs share the next lane's excl)
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const int cand = src + step;
            const uint32_t e = __shfl_sync(0xFFFFFFFFu, excl, cand & 31);
            if (cand < 32 && e <= t) src = cand;
        }
        const uint32_t s_excl = __shfl_sync(0xFFFFFFFFu, excl, src);
        const uint32_t s_o = __shfl_sync(0xFFFFFFFFu, o, src);
        const uint32_t s_item = __shfl_sync(0xFFFFFFFFu, item, src);
        const uint32_t s_bin0 = __shfl_sync(0xFFFFFFFFu, bin0, src);
        const uint32_t s_tx = __shfl_sync(0xFFFFFFFFu, tiles_x, src);
        const int s_tx0 = __shfl_sync(0xFFFFFFFFu, tx0, src);
        const int s_ty0 = __shfl_sync(0xFFFFFFFFu, ty0, src);
        const int s_wt = __shfl_sync(0xFFFFFFFFu, wt, src);
        if (t < total) {
            const uint32_t local = t - s_excl;
            const uint32_t row = local / (uint32_t)s_wt;
            const uint32_t col = local - row * (uint32_t)s_wt;
            const uint32_t pos = s_o + local;
            pkey[pos] = s_bin0 + (uint32_t)(s_ty0 + (int)row) * s_tx + (uint32_t)(s_tx0 + (int)col);
            if (emit_item != nullptr) {
                pval[pos] = pos;
                emit_item[pos] = s_item;
            } else {
                pval[pos] = s_item;
            }
        }
        if (emit_item != nullptr) {
            // the slots of the 32 pairs lie side by side (unless an item of the warp was skipped):
            // cleared by consecutive lanes
            const uint32_t pos = s_o + t - s_excl, first = __shfl_sync(0xFFFFFFFFu, pos, 0);
            const bool run = __all_sync(0xFFFFFFFFu, t >= total || pos == first + (uint32_t)lane);
            const uint32_t n = min(32u, total - t0) * kPairGradStride;
            if (run) {
                for (uint32_t q = lane; q < n; q += 32) pairgrad[(size_t)first * kPairGradStride + q] = 0.f;
            } else if (t < total) {
                for (int q = 0; q < kPairGradStride; ++q) pairgrad[(size_t)pos * kPairGradStride + q] = 0.f;
            }
        }
    }
}

// Bucket of a bin in the longest-first work order: 1023 - key, where the key
// grows with the bin's pair count (steps of 2 pairs below 1,024 pairs, of 16
// up to 9,200, one bucket above).
__device__ __forceinline__ uint32_t order_slot(uint32_t len) {
    const uint32_t key = len < 1024u ? len >> 1 : 512u + min(511u, (len - 1024u) >> 4);
    return 1023u - key;
}

// Longest-first list of work items for the persistent compositing kernels
// (list scheduling, largest job first): their work queue hands out the tiles
// with the most pairs first, so a launch does not end on a long tile taken
// late. With `halves` a bin of more than split_min pairs and more than
// 1 / split_share of all pairs becomes two items, its upper and lower half:
// one CTA walking such a list would outlast the launch's average (see
// order_spec). Where the lists are even (none longer than 7/4 of the mean) and
// `wave` CTAs run at a time, whole tiles go as far as they fill waves, and the
// last part of a wave as halves if those fit one, else whole: by their share
// of the pairs all of a few hundred tiles more than a wave would be halved,
// which ends on a third wave of halves. (Iteration of 60,000 random Gaussians
// on 1,200 tiles of 640x480: 16 x 1 tiles 304 us, all halved 336, this 284; of
// 300,000 431, 452, 384; on 1,008 tiles of three 333x251 views 380, 410, 349;
// 1,900 tiles of 800x600 463, 445, 411. On 2,400, whose last wave is more than
// half full, whole tiles 553 and halves at its end 561. Rooms, whose tiles
// differ, are not even: 1.0x.) One CTA of NT threads, a counting sort by
// bucket; items of one
// bucket come in any order (the compositing result does not depend on which CTA
// takes an item, nor on whether a tile is halved). A non-zero *cancel leaves
// the list empty.
struct OrderSpec {
    uint32_t n_bins;
    int halves;
    uint32_t split_min, split_share;
    uint32_t wave;   // CTAs that run at a time; 0: evenness is not looked at
    const uint32_t* n_pairs;
    const uint32_t* cancel;
};
template <int NT, bool EVEN>
__device__ __forceinline__ void build_work_order(const uint2* ranges, const OrderSpec& o, uint32_t* __restrict__ order) {
    constexpr int E = 1024 / NT;   // buckets a thread
    // lists a thread keeps in registers between the passes (of a launch of its own, which is a few round
    // trips to L2 long; with the evenness to look at they take one pass more)
    constexpr int R = EVEN && NT == 1024 ? 3 : 0;
    __shared__ uint32_t cnt[1024];
    __shared__ uint32_t wsum[32];
    const int t = threadIdx.x, lane = t & 31;
    uint32_t kept[R > 0 ? R : 1];
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const uint32_t b = t + u * NT;
        const uint2 r = b < o.n_bins ? __ldcg(ranges + b) : make_uint2(0u, 0u);
        kept[u] = r.y - r.x;
    }
    auto each_bin = [&](auto f) {   // f(bin, length of its list)
        if (R > 0 && o.n_bins <= (uint32_t)(R * NT)) {
#pragma unroll
            for (int u = 0; u < R; ++u)
                if (t + u * NT < o.n_bins) f(t + u * NT, kept[u]);
        } else {
            for (uint32_t b = t; b < o.n_bins; b += NT) {
                const uint2 r = __ldcg(ranges + b);   // (of this launch: past L1)
                f(b, r.y - r.x);
            }
        }
    };
    uint32_t longest = o.halves ? max(o.split_min, *o.n_pairs / o.split_share) : 0xFFFFFFFFu;
    uint32_t whole = 0xFFFFFFFFu;   // of even lists: the tiles before the halved ones
    for (int e = 0; e < E; ++e) cnt[t * E + e] = 0;
    if constexpr (EVEN) {
        __shared__ uint32_t most;
        if (t == 0) most = 0u;
        __syncthreads();
        uint32_t m = 0;
        each_bin([&](uint32_t, uint32_t len) { m = max(m, len); });
        m = __reduce_max_sync(0xFFFFFFFFu, m);
        if (lane == 0) atomicMax(&most, m);
        __syncthreads();
        if (4ull * most * o.n_bins <= 7ull * *o.n_pairs) {
            const uint32_t rest = o.n_bins % o.wave;
            whole = 2u * rest <= o.wave ? o.n_bins - rest : o.n_bins;
            longest = 0xFFFFFFFFu;
        }
    }
    __syncthreads();
    each_bin([&](uint32_t, uint32_t len) { atomicAdd(&cnt[order_slot(len)], len > longest ? 2u : 1u); });
    __syncthreads();
    uint32_t v[E], sum = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        v[e] = cnt[t * E + e];
        sum += v[e];
    }
    uint32_t x = sum;   // inclusive scan within the warp, then over the warps
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, q);
        if (lane >= q) x += y;
    }
    if (lane == 31) wsum[t >> 5] = x;
    __syncthreads();
    if (t < 32) {
        const uint32_t w = t < NT / 32 ? wsum[t] : 0u;
        uint32_t z = w;
#pragma unroll
        for (int q = 1; q < 32; q <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, z, q);
            if (lane >= q) z += y;
        }
        wsum[t] = z - w;
    }
    __syncthreads();
    uint32_t start = x - sum + wsum[t >> 5];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        cnt[t * E + e] = start;
        start += v[e];
    }
    if (EVEN && whole != 0xFFFFFFFFu) start = 2u * o.n_bins - whole;
    if (t == NT - 1) order[0] = o.cancel != nullptr && *o.cancel != 0u ? 0u : start;
    __syncthreads();
    each_bin([&](uint32_t b, uint32_t len) {
        const bool two = len > longest;
        const uint32_t p = atomicAdd(&cnt[order_slot(len)], two ? 2u : 1u);
        if (EVEN && p >= whole) {
            order[1 + 2 * p - whole] = b | (1u << kItemShift);
            order[2 + 2 * p - whole] = b | (2u << kItemShift);
        } else if (two) {
            order[1 + p] = b | (1u << kItemShift);
            order[2 + p] = b | (2u << kItemShift);
        } else {
            order[1 + p] = b;
        }
    });
}
template <bool EVEN>
__global__ void __launch_bounds__(1024) k_work_order(const uint2* __restrict__ ranges, OrderSpec spec,
                                                      uint32_t* __restrict__ order) {
    build_work_order<1024, EVEN>(ranges, spec, order);
}

// The sorted pairs' (start, end) per bin. After an overflow of the pair buffer the sorted values hold
// slots that no item wrote: every bin stays empty then, and nothing is composited. Where *fresh is set
// (a replayed iteration whose cameras are not those of the one before, which left the work list for
// them), the last CTA to finish writes the list of these ranges. Single 640x480 views of a window in
// turn, with the list of the view before: 522 us an iteration; with their own: 318.
template <bool EVEN>
__global__ void __launch_bounds__(256) k_ranges(const uint32_t* __restrict__ pkey, const uint32_t* __restrict__ P_dev,
                                                uint64_t pair_cap, uint32_t n_bins, const uint32_t* __restrict__ overflow,
                                                uint2* __restrict__ ranges, const uint32_t* __restrict__ fresh,
                                                uint32_t* __restrict__ ticket, OrderSpec spec,
                                                uint32_t* __restrict__ order) {
    if (*overflow == 0u) {
        const uint32_t P = (uint32_t)(*P_dev < pair_cap ? *P_dev : pair_cap);
        for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < P; i += gridDim.x * blockDim.x) {
            const uint32_t b = pkey[i];
            if (i == 0 || pkey[i - 1] != b) ranges[b].x = i;
            if (i == P - 1 || pkey[i + 1] != b) ranges[b].y = i + 1;
        }
    }
    if (fresh == nullptr || *fresh == 0u) return;
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x == 0) *ticket = 0u;
    build_work_order<256, EVEN>(ranges, spec, order);
}

}  // namespace

cudaError_t sort_kernels_init() {
    cudaError_t e = cudaFuncSetAttribute(k_radix_scatter<11>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(ScatterSmem<11>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_small_depth, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem));
    return e;
}

int sort_max_blocks() { return kMaxGrid; }
// Digit counts: rows of 2^8 for the pairs' blocks or of 2^11 for the depths' (a block per 2048 of the
// context's items at most), then the digits' totals. (2^11 for every block, 5 MB, made the creation of a
// context for 5,000 Gaussians 40 us longer.)
static size_t depth_blocks(int sort_blocks, size_t max_items) {
    return std::min((size_t)sort_blocks, (max_items + 2047) / 2048);
}
size_t sort_hist_words(int sort_blocks, size_t max_items) {
    return std::max((size_t)sort_blocks << 8, depth_blocks(sort_blocks, max_items) << 11) + (1u << 11);
}
static uint32_t* sort_totals(const gs_ctx* c) { return c->hist + c->hist_words - (1u << 11); }

// about 2048 elements (one scatter round) per block, each block owning one contiguous slice
static int sort_grid(const gs_ctx* c, uint32_t n_hint) {
    return (int)std::max<uint32_t>(1u, std::min<uint32_t>((uint32_t)c->sort_blocks, (n_hint + 2047u) / 2048u));
}

bool depth_sort_small(const gs_ctx* c) { return (uint64_t)c->n_views * (uint64_t)c->n <= (uint64_t)kSmallItems; }

// Raw keys in dkey[0] (and, above kSmallItems, the compacted ones in dkey[1] / dval[1]): the visible
// items in depth order to dval[0], their tile sums to tile_blocks and dcount[0].
cudaError_t sort_depth(gs_ctx* c, uint32_t n_max, uint32_t n_hint, cudaStream_t s) {
    if (depth_sort_small(c)) {
        ++c->launches;
        k_small_depth<<<1, kSmallThreads, sizeof(SmallSmem), s>>>(c->dkey[0], n_max, c->tiles_touched, c->dval[0],
                                                                 c->tile_blocks, c->dcount);
        return cudaGetLastError();
    }
    const int G = (int)std::min((size_t)sort_grid(c, n_hint), depth_blocks(c->sort_blocks, n_max));
    int cur = 1;
    for (int pass = 0; pass < 3; ++pass) {
        c->launches += G > kScanGrid ? 3 : 2;
        const cudaError_t e =
            launch_radix_pass<11>(G, c->dkey[cur], c->dval[cur], c->dkey[cur ^ 1], c->dval[cur ^ 1], c->dcount + 8, n_max,
                                  DigitSpec{c->dcount + 11, 0, pass, 3}, c->hist, sort_totals(c), s);
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    ++c->launches;
    const int blocks = (int)std::max<uint32_t>(1u, std::min<uint32_t>((n_max + 255u) / 256u, (n_hint + 255u) / 256u));
    k_item_tiles<<<blocks, 256, 0, s>>>(c->dval[0], c->tiles_touched, n_max, c->dcount + 8, c->tile_blocks,
                                         reinterpret_cast<unsigned long long*>(c->dcount));
    return cudaGetLastError();
}

cudaError_t radix_sort_pairs(gs_ctx* c, uint32_t** keys, uint32_t** vals, const uint32_t* n_dev, uint32_t n_max,
                             uint32_t n_hint, int bits, int* out_buf, cudaStream_t s) {
    int cur = 0;
    const int G = sort_grid(c, n_hint), passes = (bits + 7) / 8;
    for (int pass = 0; pass < passes; ++pass) {
        c->launches += G > kScanGrid ? 3 : 2;
        const cudaError_t e = launch_radix_pass<8>(G, keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], n_dev, n_max,
                                                   DigitSpec{nullptr, bits, pass, passes}, c->hist, sort_totals(c), s);
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    *out_buf = cur;
    return cudaSuccess;
}

cudaError_t scan_u32(gs_ctx* c, const uint32_t* in, uint32_t* out, uint32_t n, uint32_t* total_dev,
                     cudaStream_t s) {
    const int G = c->sort_blocks;
    c->launches += 2;
    k_block_sums<<<G, 256, 0, s>>>(in, n, c->hist);
    k_scan<<<G, 256, 0, s>>>(in, n, c->hist, out, total_dev);
    return cudaGetLastError();
}

// Blocks of 256 items up to which every CTA of the emission adds up the tile sums before its own, work
// that grows with their square. A 640x480 render with the sums / with a scan before it: 269 / 275 us at
// 300k Gaussians, 1,076 / 1,077 at 4M (15,625 blocks), 1,633 / 1,617 at 8M, 3,058 / 2,948 at 16M.
constexpr uint32_t kEmitSums = 16384;

cudaError_t emit_pairs(gs_ctx* c, uint32_t n_items, const uint32_t* n_dev, cudaStream_t s) {
    if (n_items == 0) return cudaSuccess;
    const uint32_t blocks = (uint32_t)(((uint64_t)n_items + 255u) / 256u);
    const bool scanned = blocks > kEmitSums;
    const uint32_t* tile_blocks = c->tile_blocks;
    if (scanned) {   // (into the depth sort's free buffer; what lies past the visible items is not read)
        cudaError_t e = scan_u32(c, c->tile_blocks, c->dkey[1], blocks, nullptr, s);
        if (e != cudaSuccess) return e;
        tile_blocks = c->dkey[1];
    }
    ++c->launches;
    k_emit<<<blocks, 256, 0, s>>>(c->dval[0], c->tiles_touched, tile_blocks, scanned, c->offsets, c->rec, c->dcam, c->n,
                                  c->tile, n_items, n_dev, (uint64_t)c->pair_cap, c->pkey[0], c->pval[0], c->dcount + 1,
                                  c->dcount + 9, c->emit_item, c->pairgrad);
    return cudaGetLastError();
}

// Deterministic mode: item k of the depth order owns the pair slots off[k] ..
// off[k] + tiles - 1 (its emission indices); a warp adds their screen gradients,
// lane l those l, l + 32, .. and then a fixed tree over the lanes, into the
// item's grad2d record. (One thread an item: a Gaussian over a thousand tiles
// was the launch's time, 65 us for 20k Gaussians in three 321x243 views; 12 us.)
__global__ void __launch_bounds__(256) k_pairgrad_reduce(const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ tiles,
                                                         const uint32_t* __restrict__ off, uint32_t n_items,
                                                         const uint32_t* __restrict__ n_dev, uint64_t pair_cap,
                                                         const float* __restrict__ pairgrad,
                                                         float* __restrict__ grad2d) {
    const int lane = threadIdx.x & 31;
    const uint32_t nv = umin(n_items, *n_dev);
    for (uint32_t k = blockIdx.x * 8 + (threadIdx.x >> 5); k < nv; k += gridDim.x * 8) {
        const uint32_t item = order[k], cnt = tiles[item];
        const uint64_t o = off[k];
        float s[kPairGradStride];
#pragma unroll
        for (int q = 0; q < kPairGradStride; ++q) s[q] = 0.f;
        if (o + cnt <= pair_cap)
            for (uint64_t e = o + lane; e < o + cnt; e += 32)
#pragma unroll
                for (int q = 0; q < kPairGradStride; ++q) s[q] += pairgrad[e * kPairGradStride + q];
        float v = 0.f;
#pragma unroll
        for (int q = 0; q < kPairGradStride; ++q) {
            float t = s[q];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
            if (lane == q) v = t;
        }
        if (lane < kPairGradStride) grad2d[(size_t)item * kGrad2dStride + lane] = v;
    }
}

cudaError_t reduce_pair_grads(gs_ctx* c, cudaStream_t s) {
    const uint32_t items = (uint32_t)c->n_views * (uint32_t)c->n;
    if (c->pairgrad == nullptr || items == 0) return cudaSuccess;
    ++c->launches;
    const int grid = (int)std::min<uint32_t>((items + 7) / 8, (uint32_t)c->num_sms * 8);
    k_pairgrad_reduce<<<grid, 256, 0, s>>>(c->dval[0], c->tiles_touched, c->offsets, items,
                                                          c->dcount + 8, (uint64_t)c->pair_cap, c->pairgrad,
                                                          c->grad2d);
    return cudaGetLastError();
}

static OrderSpec order_spec(const gs_ctx* c) {
    // The 16 x 2 layout runs 6 CTAs an SM. With no more halves than that in all, every tile is
    // halved: a CTA's chain of dependent visits is the launch's time, and one pixel a thread instead
    // of two shortens it (160x120 with 2k Gaussians: fused kernel 57 -> 29 us). Otherwise a bin is
    // halved that holds more than half an average CTA's pairs (all pairs over 12 CTAs an SM); lower,
    // the halves' second staging of the list costs more than the balance gives (fused kernel at 9, 12
    // and 18 an SM: 1200x680 keyframe with 300k 372, 341, 320 us and 527 without halves; one with
    // lists of similar length 337, 343, 354 us; 8 x 640x480 window 782, 785, 797 us). Bins of 128
    // pairs or less take a CTA no longer than the launch's other latencies.
    OrderSpec o;
    o.n_bins = (uint32_t)c->n_bins;
    o.halves = half_tiles(c) ? 1 : 0;
    const int wave = 6 * c->num_sms;
    const bool all = 2 * (int64_t)c->n_bins <= wave;
    o.split_min = all ? 0u : 128u;
    o.split_share = all ? 0xFFFFFFFFu : 12u * (uint32_t)c->num_sms;
    o.wave = o.halves && c->n_bins >= wave && c->n_bins <= 3 * wave ? (uint32_t)wave : 0u;
    o.n_pairs = c->dcount;
    // a render with an unreported non-finite value is not made (a replay's order is for the next one)
    o.cancel = c->order_ahead ? nullptr : c->dcount + 10;
    return o;
}

cudaError_t compute_ranges(gs_ctx* c, cudaStream_t s) {
    // (a mapping iteration zeroes the ranges on its side stream)
    if (!c->side_zeroed) cudaMemsetAsync(c->ranges, 0, sizeof(uint2) * (size_t)c->n_bins, s);
    ++c->launches;
    const OrderSpec spec = order_spec(c);
    auto ranges = spec.wave != 0u ? k_ranges<true> : k_ranges<false>;
    ranges<<<c->num_sms * 8, 256, 0, s>>>(c->pkey[c->pair_buf], c->dcount, (uint64_t)c->pair_cap, (uint32_t)c->n_bins,
                                          c->dcount + 9, c->ranges, c->order_ahead ? c->dcount + 13 : nullptr,
                                          c->dcount + 14, spec, c->work_order);
    if (c->points != nullptr) return launch_point_items(c, *c->points, true, s);
    return c->order_ahead ? cudaGetLastError() : launch_work_order(c, s);
}

cudaError_t launch_work_order(gs_ctx* c, cudaStream_t s) {
    ++c->launches;
    const OrderSpec spec = order_spec(c);
    auto work_order = spec.wave != 0u ? k_work_order<true> : k_work_order<false>;
    work_order<<<1, 1024, 0, s>>>(c->ranges, spec, c->work_order);
    return cudaGetLastError();
}

}  // namespace gs

// ---------------------------------------------------------------------------
// Allocation-free variant of the pair sort, for callers that must not allocate
// device memory (for example code that runs while another component owns the
// device allocator, or a real-time loop that forbids cudaMalloc). Its scratch
// is one file-scope __device__ array that every GPU loading this library holds
// until the process exits.

namespace gs {
namespace {

constexpr uint32_t kStaticSortMaxPairs = 1u << 20;                       // largest n accepted
constexpr int kStaticSortMaxBlocks = (int)((kStaticSortMaxPairs + 4095u) / 4096u);
static_assert(kStaticSortMaxBlocks <= kMaxGrid, "blocks that the digit scan takes");
constexpr size_t kStaticSortWords = 64                                  // [0] count sentinel
                                    + 2 * (size_t)kStaticSortMaxPairs    // ping-pong keys and values
                                    + 256 * (size_t)kStaticSortMaxBlocks + 256;   // histograms, digit totals
static __device__ __align__(256) uint32_t g_static_sort_scratch[kStaticSortWords];

// [a, a + n) and [b, b + n) words overlap
bool ranges_overlap(const void* a, const void* b, uint64_t n) {
    const uint64_t x = (uint64_t)(uintptr_t)a, y = (uint64_t)(uintptr_t)b, len = 4 * n;
    return x < y + len && y < x + len;
}

}  // namespace
}  // namespace gs

extern "C" int gs_sort_pairs_static(const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out,
                                    uint32_t* vals_out, int64_t n, int bits, void* stream) {
    using namespace gs;
    if (n < 0 || bits < 1 || bits > 32) return GS_ERR_ARG;
    if (n > (int64_t)kStaticSortMaxPairs) return GS_ERR_CAPACITY;
    if (n == 0) return GS_OK;
    if (!keys_in || !vals_in || !keys_out || !vals_out) return GS_ERR_ARG;
    // a pass reads the inputs while it writes the outputs: no output may overlap an input or the
    // other output (the inputs may overlap each other)
    const uint64_t un64 = (uint64_t)n;
    if (ranges_overlap(keys_out, vals_out, un64) || ranges_overlap(keys_out, keys_in, un64) ||
        ranges_overlap(keys_out, vals_in, un64) || ranges_overlap(vals_out, keys_in, un64) ||
        ranges_overlap(vals_out, vals_in, un64))
        return GS_ERR_ARG;
    // an unchecked error of earlier work is left for its owner: nothing is launched
    if (cudaPeekAtLastError() != cudaSuccess) return GS_ERR_CUDA;
    // The device address of the scratch array on the current device. In host code the array's
    // name is only a host-side stand-in; the runtime maps it to this device's copy. Resolved on
    // every call (a lookup once the device code is loaded, which the first call on a device
    // does), so a context that was reset and re-created gets its own address.
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_sort_scratch) != cudaSuccess || p == nullptr) {
        cudaGetLastError();   // this call's own error, reported by the return code
        return GS_ERR_CUDA;
    }
    uint32_t* base = static_cast<uint32_t*>(p);
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t* sentinel = base;
    uint32_t* tmp_k = base + 64;
    uint32_t* tmp_v = tmp_k + kStaticSortMaxPairs;
    uint32_t* hist = tmp_v + kStaticSortMaxPairs;
    const uint32_t un = (uint32_t)n;
    const int G = (int)std::max<uint32_t>(1u, std::min<uint32_t>((uint32_t)kStaticSortMaxBlocks, (un + 4095u) / 4096u));
    uint32_t* dtot = hist + (size_t)256 * G;
    // the count is passed as n_max with a device-side bound of 0xFFFFFFFF
    if (cudaMemsetAsync(sentinel, 0xFF, sizeof(uint32_t), s) != cudaSuccess) {
        cudaGetLastError();
        return GS_ERR_CUDA;
    }
    const int passes = (bits + 7) / 8;
    const uint32_t* src_k = keys_in;
    const uint32_t* src_v = vals_in;
    for (int i = 0; i < passes; ++i) {
        // destinations alternate so that the last pass writes the caller's output
        const bool to_out = ((passes - i) & 1) == 1;
        uint32_t* dk = to_out ? keys_out : tmp_k;
        uint32_t* dv = to_out ? vals_out : tmp_v;
        if (launch_radix_pass<8>(G, src_k, src_v, dk, dv, sentinel, un, DigitSpec{nullptr, bits, i, passes}, hist, dtot, s) !=
            cudaSuccess)
            return GS_ERR_CUDA;
        src_k = dk;
        src_v = dv;
    }
    return GS_OK;
}
