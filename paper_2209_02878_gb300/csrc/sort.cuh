// Stable LSD radix sort of (key, value) pairs on the device, 8-bit digits,
// used for the triangle Morton keys (a3) and for the coherent segment order.
//
// One pass over digit `shift`:
//   k_sort_hist    per tile (radix_sort): digit histogram -> hist[d][tile]
//   k_sort_scan    one block per digit: exclusive scan over the tiles of
//                  hist[d][*] in place, digit total -> totals[d]
//   k_sort_scatter per tile: digit bases (exclusive scan of totals), stable
//                  rank within the tile (each warp owns a contiguous run and
//                  ranks equal digits with __match_any_sync in key order),
//                  scatter to base + tile offset + rank.
// With at most kSortFuseTiles tiles the scan kernel is skipped: every
// scatter block sums the (few) tile histograms of its digit itself.  Tiles hold
// 1,024 keys, those of large sorts 2,048 (radix_sort).
//
// What bounds the scatter is its stores: 35 us a pass at 1.31M 12-byte entries
// when each lane stores to its own sector, 22 when the tile is ordered by digit
// in shared memory first (and 16 either way where the digits are already
// nearly in order).  The build of that mesh as a graph: 434 -> 359 us with the
// box pass's whole-sector stores and the kept centroids (build.cu); the order
// of 1,000,003 segments 100 -> 74 us, of 262,144 96 -> 43 us, of 65,536 62 -> 35.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rsi_internal.cuh"

namespace rsi {

template <typename K, int ITEMS>
__global__ void __launch_bounds__(kSortThreads) k_sort_hist(const K* __restrict__ keys, int n,
                                                            int shift, uint32_t* __restrict__ hist,
                                                            int ntiles) {
    __shared__ uint32_t h[kSortBins];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * kSortThreads * ITEMS;
    uint32_t dig[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int pos = base + it * kSortThreads + threadIdx.x;
        dig[it] = pos < n ? (uint32_t)(keys[pos] >> shift) & 0xffu : kSortBins;
    }
#pragma unroll
    for (int it = 0; it < ITEMS; ++it)
        if (dig[it] < kSortBins) atomicAdd(&h[dig[it]], 1u);
    __syncthreads();
    hist[threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Block-wide exclusive scan of one value per thread (blockDim.x <= 1024).
__device__ __forceinline__ uint32_t block_scan_u32(uint32_t x, uint32_t* total) {
    __shared__ uint32_t ws[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        uint32_t v = lane < nw ? ws[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        ws[lane] = v;
    }
    __syncthreads();
    if (total) *total = ws[(blockDim.x >> 5) - 1];
    const uint32_t r = incl - x + (w > 0 ? ws[w - 1] : 0u);
    __syncthreads();
    return r;
}

// One block (256 threads) per digit: exclusive scan of hist[d][0..ntiles).
static __global__ void __launch_bounds__(256) k_sort_scan(uint32_t* __restrict__ hist, int ntiles,
                                                   uint32_t* __restrict__ totals) {
    uint32_t* row = hist + (size_t)blockIdx.x * ntiles;
    const int per = (ntiles + blockDim.x - 1) / blockDim.x;
    const int b = threadIdx.x * per, e = min(ntiles, b + per);
    uint32_t sum = 0;
    for (int q = b; q < e; ++q) sum += row[q];
    uint32_t tot;
    uint32_t run = block_scan_u32(sum, &tot);
    for (int q = b; q < e; ++q) {
        const uint32_t x = row[q];
        row[q] = run;
        run += x;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = tot;
}

// The sums read the histograms a row per thread.  us of a build (of a segment
// order) as a graph, folded in / with the scan kernel, by tiles: 16: 55.7 / 56.9
// (26.5 / 29.3), 20: 54.8 / 58.6 (26.6 / 32.3), 28: 58.7 / 60.1 (29.3 / 32.2), 32:
// 69.7 / 59.5 (41.2 / 33.0), 36: 61.4 / 59.8 (31.5 / 32.8), 48: 73.1 / 62.5 (41.3 /
// 32.5), 64: 89.2 / 63.3 (57.4 / 33.0): from 32 on the multiples of 16 tiles, whose
// rows lie a multiple of 64 B apart, are the slowest.  (Tile-major histograms, whose reads coalesce:
// build of 30 tiles 69.8 against 64.5.)
constexpr int kSortFuseTiles = 31;

template <typename K, int ITEMS, bool FUSED>
__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(
    const K* __restrict__ kin, const uint32_t* __restrict__ vin, K* __restrict__ kout,
    uint32_t* __restrict__ vout, int n, int shift, const uint32_t* __restrict__ hist,
    const uint32_t* __restrict__ totals, int ntiles) {
    constexpr int W = kSortThreads / 32;
    // Large sorts order the tile by digit in shared memory first, so that a
    // warp's stores run along a few output runs instead of touching a sector
    // per lane.
    constexpr bool REORDER = ITEMS > 4;
    __shared__ uint32_t cnt[W][kSortBins];
    __shared__ K sk[REORDER ? kSortThreads * ITEMS : 1];
    __shared__ uint32_t sv[REORDER ? kSortThreads * ITEMS : 1];
    __shared__ uint32_t gbase[REORDER ? kSortBins : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int q = threadIdx.x; q < W * kSortBins; q += kSortThreads) (&cnt[0][0])[q] = 0;
    // this tile's offset within digit d (FUSED: summed here from the raw tile
    // histograms) and the digit total; kSortThreads == bins, thread = digit
    uint32_t toff, dtot;
    if (FUSED) {
        const uint32_t* row = hist + (size_t)threadIdx.x * ntiles;
        toff = dtot = 0u;
        for (int q = 0; q < ntiles; ++q) {
            const uint32_t x = row[q];
            toff += q < (int)blockIdx.x ? x : 0u;
            dtot += x;
        }
    } else {
        toff = hist[threadIdx.x * ntiles + blockIdx.x];
        dtot = totals[threadIdx.x];
    }
    // digit base = exclusive scan of the digit totals
    const uint32_t dbase = block_scan_u32(dtot, nullptr);
    const int wbase = blockIdx.x * (kSortThreads * ITEMS) + w * (32 * ITEMS);
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t local[ITEMS];
    K key[ITEMS];
    uint32_t val[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int pos = wbase + it * 32 + lane;
        key[it] = pos < n ? kin[pos] : (K)0;
        val[it] = pos < n ? vin[pos] : 0u;
    }
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const bool valid = wbase + it * 32 + lane < n;
        const uint32_t d = valid ? ((uint32_t)(key[it] >> shift) & 0xffu) : 0x100u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t rank = __popc(peers & lt);
        const uint32_t c = valid ? cnt[w][d] : 0u;
        __syncwarp();
        if (valid && rank == 0) cnt[w][d] = c + __popc(peers);
        __syncwarp();
        local[it] = c + rank;
    }
    __syncthreads();
    // this tile's keys of digit d, by warp, and (REORDER) where digit d starts
    // in the tile
    const int d0 = threadIdx.x;
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < W; ++q) mine += cnt[q][d0];
    uint32_t run = dbase + toff;
    if (REORDER) {
        const uint32_t start = block_scan_u32(mine, nullptr);
        gbase[d0] = run - start;  // global position of digit d0's run less its local one
        run = start;
    }
#pragma unroll
    for (int q = 0; q < W; ++q) {
        const uint32_t x = cnt[q][d0];
        cnt[q][d0] = run;
        run += x;
    }
    __syncthreads();
    if (!REORDER) {
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            if (wbase + it * 32 + lane < n) {
                const uint32_t d = (uint32_t)(key[it] >> shift) & 0xffu;
                const uint32_t o = cnt[w][d] + local[it];
                kout[o] = key[it];
                vout[o] = val[it];
            }
        }
        return;
    }
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        if (wbase + it * 32 + lane < n) {
            const uint32_t d = (uint32_t)(key[it] >> shift) & 0xffu;
            const uint32_t o = cnt[w][d] + local[it];
            sk[o] = key[it];
            sv[o] = val[it];
        }
    }
    __syncthreads();
    const int have = min(n - (int)blockIdx.x * (kSortThreads * ITEMS), kSortThreads * ITEMS);
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int p = it * kSortThreads + threadIdx.x;
        if (p < have) {
            const K k = sk[p];
            const uint32_t o = gbase[(uint32_t)(k >> shift) & 0xffu] + (uint32_t)p;
            kout[o] = k;
            vout[o] = sv[p];
        }
    }
}

// Sort keys[0] / vals[0] (n entries) over the digits at `shifts`; buffers
// keys[1] / vals[1] are ping-pong space; *out receives the index of the
// buffer pair holding the result.  Tiles hold 1024 keys below 2^18 keys (more
// blocks for small sorts: from 2^17 on, the build of 131,072 triangles takes 83
// us instead of 78), 2048 above (4096: 362 against 359 us at 1.31M).  hist:
// kSortBins * ceil(n / 1024) words, totals: kSortBins words.
template <typename K, int ITEMS>
static cudaError_t radix_sort_tiles(K* keys[2], uint32_t* vals[2], int n, const int* shifts,
                                    int np, uint32_t* hist, uint32_t* totals, cudaStream_t s,
                                    int* out) {
    const int tile = kSortThreads * ITEMS;
    const int ntiles = (n + tile - 1) / tile;
    int cur = 0;
    for (int p = 0; p < np && n > 0; ++p) {
        k_sort_hist<K, ITEMS><<<ntiles, kSortThreads, 0, s>>>(keys[cur], n, shifts[p], hist,
                                                              ntiles);
        auto scatter = k_sort_scatter<K, ITEMS, false>;
        if (ITEMS <= 4 && ntiles <= kSortFuseTiles)  // large sorts always have more tiles
            scatter = k_sort_scatter<K, ITEMS <= 4 ? ITEMS : 4, true>;
        else
            k_sort_scan<<<kSortBins, 256, 0, s>>>(hist, ntiles, totals);
        scatter<<<ntiles, kSortThreads, 0, s>>>(keys[cur], vals[cur], keys[1 - cur],
                                                vals[1 - cur], n, shifts[p], hist, totals, ntiles);
        cur = 1 - cur;
    }
    *out = cur;
    return cudaGetLastError();
}

template <typename K>
cudaError_t radix_sort(K* keys[2], uint32_t* vals[2], int n, const int* shifts, int np,
                       uint32_t* hist, uint32_t* totals, cudaStream_t s, int* out) {
    if (n < (1 << 18))
        return radix_sort_tiles<K, 4>(keys, vals, n, shifts, np, hist, totals, s, out);
    return radix_sort_tiles<K, kSortItems>(keys, vals, n, shifts, np, hist, totals, s, out);
}

}  // namespace rsi
