// Kernels of the phased traversal loop (walk.cuh) over one mesh.
#include <cuda_runtime.h>

#include "rsi_trace.h"
#include "walk.cuh"

namespace rsi {

// SMALL: few enough segments for one set-up batch per resident warp.  They are
// dealt out evenly (f to each warp) instead of being taken from the counter:
// warps with fewer segments diverge less, which is what bounds the smallest
// launches (10,000 segments over 1,922 triangles 53 -> 35 us), and the
// triangle tests do not wait for lanes that a refill would have filled.
template <int MODE, bool STATS, bool LEAFN, bool SMALL>
__global__ void __maxnreg__(kWalkRegs<MODE>) k_walk(TraceParams P) {
    extern __shared__ float4 stage4[];
    TraceCtx C;
    C.A = P.A;
    C.B = P.B;
    C.nR = P.nR;
    C.nodes = P.nodes;
    C.qnodes = P.qnodes;
    C.frame = P.frame;
    C.coarse = P.nT > 0 && walk_coarse(*P.coarse, P.nT);
    C.tris = P.tris;
    C.max_visits = P.max_visits;
    C.fetch = P.fetch;
    C.ready = P.ready;
    C.ready_chunk = P.ready_chunk;
    C.wait_polls = P.wait_polls > 0 ? P.wait_polls : kWaitPolls;
    C.order = P.order;
    C.status = P.status;
    C.out = P.out;
    TravStats st = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
    unsigned long long segs = 0;
    using Stage = WalkStage<kOwn<MODE>>;
    Stage& sg = ((Stage*)stage4)[threadIdx.x >> 5];
    if (SMALL) {
        const int64_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        const int64_t lo = min(P.nR, w * P.fetch);
        walk_loop<MODE, STATS, LEAFN, kOwn<MODE>>(C, sg, P.root, (unsigned)lo,
                                      (unsigned)min(P.nR, lo + P.fetch), false, WalkNone{}, st,
                                      segs);
    } else {
        walk_loop<MODE, STATS, LEAFN, kOwn<MODE>>(C, sg, P.root, 0u, 0u, true, WalkCounter{C, P.walk_work}, st,
                                      segs);
        walk_finish(P.walk_work);
    }
    if (STATS) flush_stats(st, P.stats, segs);
}

template <bool STATS, bool LEAFN, bool SMALL>
static WalkFn pick_walk(int mode) {
    if (mode == RSI_MODE_BOOL) return k_walk<RSI_MODE_BOOL, STATS, LEAFN, SMALL>;
    if (mode == RSI_MODE_COUNT) return k_walk<RSI_MODE_COUNT, STATS, LEAFN, SMALL>;
    return k_walk<RSI_MODE_NEAREST, STATS, LEAFN, SMALL>;
}

WalkFn walk_kernel(int mode, bool stats, bool leafn, bool small) {
    if (stats) return leafn ? pick_walk<true, true, false>(mode) : pick_walk<true, false, false>(mode);
    if (small) return leafn ? pick_walk<false, true, true>(mode) : pick_walk<false, false, true>(mode);
    return leafn ? pick_walk<false, true, false>(mode) : pick_walk<false, false, false>(mode);
}

// Dynamic shared memory of a block.
int walk_smem(int mode, int block) {
    return block / 32 * (int)(mode == RSI_MODE_NEAREST ? sizeof(WalkStage<kOwn<RSI_MODE_NEAREST>>)
                                                        : sizeof(WalkStage<kOwn<RSI_MODE_BOOL>>));
}

// 64-bit segment indices, and leaf references that do not fit an item (leaf
// sizes above 1 from 2^28 triangles on), stay with the general loop.
bool walk_fits(int64_t nR, int64_t n, int leaf_size) {
    return nR < (int64_t)1 << 31 && (leaf_size == 1 || n < (int64_t)1 << 28);
}

// First item of every segment's walk over a mesh of n triangles at offset
// off: the Karras root's slot (not the root slot above it, whose only use is
// the box of the whole mesh: 9.0 -> 8.0 visits per segment of the paper-scale
// query), or the mesh as one leaf.
int walk_start(int off, int n, int leaf_size) {
    if (n == 0) return kNoRoot;
    if (n > leaf_size) return off;
    return leaf_size > 1 ? ~((off << 3) | (n - 1)) : ~off;
}

}  // namespace rsi
