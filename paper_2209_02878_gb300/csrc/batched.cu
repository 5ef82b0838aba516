// Batched traversal: many independent (mesh, segments, mode) problems in one
// persistent launch per mode.  The work is a list of tiles (a few hundred segments
// of one item) ordered by decreasing estimated cost per segment (log2 N_t,
// NEAREST and COUNT weighted above BOOL) so the expensive tiles start first;
// each warp pulls the next tile from one atomic counter and runs the same
// per-lane refill traversal as the single-mesh kernel over the tile, in that
// item's mode.  All meshes live in one concatenated node / triangle storage
// built by one multi-mesh build.
#include <cuda_runtime.h>

#include "rsi_trace.h"
#include "walk.cuh"

namespace rsi {

// All three modes are inlined into one kernel; without a cap it needs ~170
// registers (two warps per scheduler).  128 measured fastest on the 64-mesh
// mix (8.37 ms against 8.79 ms at 96 and 9.52 ms at 72, where the nearest
// path spills).
template <int STACK>
__global__ void __maxnreg__(128) k_batch(BatchParams P) {
    TravStats st = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
    unsigned long long segs = 0;
    const int lane = threadIdx.x & 31;
    while (true) {
        unsigned long long t = 0ull;
        if (lane == 0) t = atomicAdd(P.work, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= (unsigned long long)P.n_tiles) break;
        const BatchTile tile = P.tiles[t];
        const BatchItemDev& it = P.items[tile.item];
        TraceCtx C;
        C.A = it.A;
        C.B = it.B;
        C.nR = it.nR;
        C.root = it.root;
        C.root4 = it.root;
        C.nodes = P.nodes;
        C.nodes4 = P.nodes4;
        C.tris = P.tris;
        C.treelet = nullptr;
        C.snodes = nullptr;
        C.S = 0;
        C.max_visits = P.max_visits;
        C.fetch = kFetchChunk;  // unused: each tile is one warp's whole pool
        C.ready = nullptr;
        C.ready_chunk = 1;
        C.wait_polls = kWaitPolls;
        C.order = nullptr;
        C.status = P.status;
        C.out = it.out;
        switch (it.mode) {
            case RSI_MODE_BOOL:
                trace_loop<RSI_MODE_BOOL, STACK, false, 2, false>(C, nullptr, tile.lo, tile.hi, st,
                                                                  segs);
                break;
            case RSI_MODE_COUNT:
                trace_loop<RSI_MODE_COUNT, STACK, false, 2, false>(C, nullptr, tile.lo, tile.hi, st,
                                                                   segs);
                break;
            default:
                trace_loop<RSI_MODE_NEAREST, STACK, false, 2, false>(C, nullptr, tile.lo, tile.hi,
                                                                     st, segs);
                break;
        }
    }
}

// The phased loop (walk.cuh), for the default stack: one kernel per mode over
// that mode's tiles, so that each keeps its own register count.  Inlined into
// one kernel the three need 128 registers: 1,790 us on 16 meshes with 3.5M
// segments, and 2,178 us out of line (the calls save too much); the general
// loop, inlined at 128, 2,265 us; side by side at 80 registers with tiles of
// 1,024, each run dry, 1,549; as below 1,143.
//
// A warp goes on with the tiles of one item (they are consecutive in the list)
// without letting its lanes run dry in between; a tile of another item waits
// until they have finished.
template <int MODE, bool LEAFN>
__global__ void __maxnreg__(kBatchRegs) k_batch_walk(BatchParams P) {
    extern __shared__ float4 stage4[];
    WalkStage<false>& sg = ((WalkStage<false>*)stage4)[threadIdx.x >> 5];
    TravStats st = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
    unsigned long long segs = 0;
    const BatchTile* tiles = P.tiles + P.mode_first[MODE];
    const unsigned n = (unsigned)P.mode_tiles[MODE];
    auto take = [&]() {  // index of the next tile, warp-uniform
        unsigned t = 0u;
        if ((threadIdx.x & 31) == 0) t = (unsigned)atomicAdd(P.work + MODE, 1ull);
        return __shfl_sync(0xffffffffu, t, 0);
    };
    TraceCtx C;
    C.nodes = P.nodes;
    C.qnodes = P.qnodes;
    C.tris = P.tris;
    C.max_visits = P.max_visits;
    C.ready = nullptr;
    C.order = nullptr;
    C.status = P.status;
    unsigned t = take();
    while (t < n) {
        const BatchTile tile = tiles[t];
        const BatchItemDev& it = P.items[tile.item];
        C.A = it.A;
        C.B = it.B;
        C.nR = it.nR;
        C.out = it.out;
        C.frame = P.frame + 2 * tile.item;
        C.coarse = it.n > 0 && walk_coarse(P.coarse[tile.item], it.n);
        auto next = [&](unsigned& pool, unsigned& pool_end) {
            t = take();
            if (t >= n || tiles[t].item != tile.item) return false;
            pool = (unsigned)tiles[t].lo;
            pool_end = (unsigned)tiles[t].hi;
            return true;
        };
        walk_loop<MODE, false, LEAFN, false>(C, sg, it.start, (unsigned)tile.lo, (unsigned)tile.hi, true,
                                      next, st, segs);
    }
}

using BatchFn = void (*)(BatchParams);
static BatchFn batch_walk_kernel(int mode, bool leafn) {
    if (mode == RSI_MODE_BOOL)
        return leafn ? k_batch_walk<RSI_MODE_BOOL, true> : k_batch_walk<RSI_MODE_BOOL, false>;
    if (mode == RSI_MODE_COUNT)
        return leafn ? k_batch_walk<RSI_MODE_COUNT, true> : k_batch_walk<RSI_MODE_COUNT, false>;
    return leafn ? k_batch_walk<RSI_MODE_NEAREST, true> : k_batch_walk<RSI_MODE_NEAREST, false>;
}

// Zero the work counters and the compaction counters of the items that compact.
__global__ void k_zero_counts(const BatchItemDev* items, int n, unsigned long long* work) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < 3) work[k] = 0ull;
    if (k < n && items[k].out.hit_idx) *items[k].out.n_hits = 0;
}

const void* batch_kernel(int stack) {
    switch (stack) {
        case 8: return (const void*)k_batch<8>;
        case 32: return (const void*)k_batch<32>;
        default: return (const void*)k_batch<64>;
    }
}

static int batch_grid(int64_t n_tiles, int block, int grid) {
    const int64_t need = (n_tiles + block / 32 - 1) / (block / 32);
    return need < grid ? (int)need : grid;
}

// The modes run side by side (fork / join on aux streams): each grid fills the
// device, so the blocks of the next mode start as those of the one before
// run out of tiles.
static cudaError_t launch_batch_walk(const BatchParams& P, int block, cudaStream_t s,
                                     const BatchFork& fk) {
    int used = 0;  // modes launched so far; the first stays on s
    for (int mode = 2; mode >= 0; --mode) {  // NEAREST, the dearest, first
        if (P.mode_tiles[mode] == 0) continue;
        BatchFn fn = batch_walk_kernel(mode, P.leaf_size > 1);
        const int bl = max_block((const void*)fn, block);
        const int smem = (bl / 32) * (int)sizeof(WalkStage<false>);
        int grid = 0;
        cudaError_t e = occupancy_grid((const void*)fn, bl, smem, &grid);
        if (e != cudaSuccess) return e;
        cudaStream_t q = s;
        if (used > 0) {
            q = fk.aux[used - 1];
            e = cudaStreamWaitEvent(q, fk.start, 0);
            if (e != cudaSuccess) return e;
        } else {
            e = cudaEventRecord(fk.start, s);
            if (e != cudaSuccess) return e;
        }
        fn<<<batch_grid(P.mode_tiles[mode], bl, grid), bl, smem, q>>>(P);
        e = cudaGetLastError();
        if (used > 0) {  // join even when the launch failed: s must not run ahead
            cudaError_t j = cudaEventRecord(fk.done[used - 1], q);
            if (j == cudaSuccess) j = cudaStreamWaitEvent(s, fk.done[used - 1], 0);
            if (e == cudaSuccess) e = j;
        }
        if (e != cudaSuccess) return e;
        ++used;
    }
    return cudaSuccess;
}

cudaError_t launch_batch(const BatchParams& P, int block, int stack, cudaStream_t s,
                         const BatchFork& fk) {
    if (P.n_tiles == 0) return cudaSuccess;
    k_zero_counts<<<(P.n_items + 255) / 256, 256, 0, s>>>(P.items, P.n_items, P.work);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (P.walk && stack == 64) return launch_batch_walk(P, block, s, fk);
    const void* fn = batch_kernel(stack);
    block = max_block(fn, block);
    int grid = 0;
    e = occupancy_grid(fn, block, 0, &grid);
    if (e != cudaSuccess) return e;
    grid = batch_grid(P.n_tiles, block, grid);
    switch (stack) {
        case 8: k_batch<8><<<grid, block, 0, s>>>(P); break;
        case 32: k_batch<32><<<grid, block, 0, s>>>(P); break;
        default: k_batch<64><<<grid, block, 0, s>>>(P); break;
    }
    return cudaGetLastError();
}

}  // namespace rsi
