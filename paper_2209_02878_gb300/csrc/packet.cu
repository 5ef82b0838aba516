// Warp-cooperative ("packet") traversal, the alternative to one stack per
// segment for coherent segments (the divergence remark of Sec. 4.1 on
// Morton-sorted rays; launch option `packet`).
//
// A warp takes 32 consecutive segments in processing order (input order, or
// the coherent order of sort_bits) and walks the tree once for all of them:
//  - every node is fetched once per warp (all lanes load the same record, a
//    broadcast), and each lane slab-tests its own segment against the two
//    child boxes;
//  - each lane tests the triangles of the leaves its own segment enters
//    (BOOL lanes stop at their first crossing, NEAREST lanes shrink their own
//    t limit);
//  - the warp descends into a child when any active lane enters it, the near
//    child first by majority vote of the lanes entering both, and keeps the
//    other on one warp-uniform stack (held by every lane at the same index,
//    so its local-memory accesses are coalesced);
//  - the warp stops when the stack is empty or no lane is active.
// The nodes, the box test and the triangle test are those of the phased loop
// (walk.cuh).  The results are the per-segment results (the same leaf tests, in a
// different order); the cost is the union of the 32 paths, so it pays off
// only when a warp's segments are close in space and direction.
#include <cuda_runtime.h>

#include "rsi_trace.h"
#include "walk.cuh"

namespace rsi {

constexpr int kPacketBlock = 128;

template <int MODE>
struct PacketRegs {
    static constexpr int value = MODE == RSI_MODE_NEAREST ? 80 : 72;
};

template <int MODE, bool STATS, bool LEAFN, bool COARSE>
__device__ __forceinline__ void packet_loop(const TraceCtx& C, int start, unsigned long long* work,
                                            TravStats& st, unsigned long long& segs) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int stack[kWalkStack + 1];
    stack[0] = kDone;
    while (true) {
        unsigned long long b = 0ull;
        if (lane == 0) b = atomicAdd(work, 32ull);
        b = __shfl_sync(FULL, b, 0);
        if (b >= (unsigned long long)C.nR) break;
        const int64_t pos = (int64_t)b + lane;
        bool valid = pos < C.nR;
        int64_t i = pos;
        if (valid && C.order) {  // a caller's order: entries outside [0, nR) are skipped
            i = C.order[pos];
            if (i < 0 || i >= C.nR) {
                atomicCAS(C.status, 0, RSI_ERR_BAD_INDEX);
                valid = false;
            }
        }
        if (!valid) i = 0;
        WalkSeg s;
        int count = 0;
        unsigned best = kNoBest;
        float tlo = 0.f, tlim = 1.f;
        bool act = false;
        if (valid) {
            if (STATS) ++segs;
            act = walk_setup(C, i, s) && start != kNoRoot;
            s.select();
            s.range();
        }
        s.swap = 0u;  // every lane reads the same half first (idle lanes read it too)
        int item = start, sp = 0, visits = 0;  // the stack is the warp's: the same in every lane
        while (__ballot_sync(FULL, act)) {
            if (++visits > C.max_visits) {  // warp-uniform: a corrupt tree
                if (lane == 0) atomicCAS(C.status, 0, RSI_ERR_INTERNAL);
                break;
            }
            if (item < 0) {  // a mesh that is one leaf
                if (act)
                    walk_leaf<MODE, STATS, LEAFN>(C, s, i, item, count, best, tlo, tlim, st);
                break;
            }
            constexpr int K = COARSE ? 2 : 4;
            bool h[K];
            float t[K];
            int x[K];
            if (STATS && act) ++st.visits;
            if constexpr (COARSE)
                walk_node2<MODE == RSI_MODE_NEAREST, LEAFN>(C, s, item, tlim, h, t, x);
            else
                walk_node4<MODE == RSI_MODE_NEAREST>(C, s, item, tlim, h, t, x);
            unsigned leaves = 0u;  // children that are leaves some lane enters
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (x[k] < 0 && __ballot_sync(FULL, act && h[k])) leaves |= 1u << k;
            while (leaves) {
                const int k = __ffs(leaves) - 1;
                leaves &= leaves - 1u;
                int xk = x[0];
                bool hk = h[0];
#pragma unroll
                for (int q = 1; q < K; ++q)
                    if (k == q) {
                        xk = x[q];
                        hk = h[q];
                    }
                if (act && hk &&
                    walk_leaf<MODE, STATS, LEAFN>(C, s, i, xk, count, best, tlo, tlim, st))
                    act = false;  // BOOL: the first crossing decides
            }
            // descend into the child that most lanes enter first, push the others
            int kb = -1;
            float tb = 2.f;
            unsigned m[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const bool g = act && h[k] && x[k] >= 0;
                m[k] = __ballot_sync(FULL, g);
                if (g && t[k] < tb) {
                    tb = t[k];
                    kb = k;
                }
            }
            int first = -1, votes = -1, next = kDone;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int v = __popc(__ballot_sync(FULL, kb == k));
                if (m[k] && v > votes) {
                    votes = v;
                    first = k;
                    next = x[k];
                }
            }
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (m[k] && k != first) walk_push(stack, sp, x[k]);
            item = first >= 0 ? next : stack[sp--];
            if (item == kDone) break;
        }
        float dist = 0.f, Pt[3] = {0.f, 0.f, 0.f};
        Result res;
        if (valid) {
            if (MODE == RSI_MODE_BOOL) {
                C.out.flag[i] = (uint8_t)(count > 0);
            } else if (MODE == RSI_MODE_COUNT) {
                C.out.count[i] = count;
            } else {
                walk_nearest_out<STATS>(C, s, i, best, dist, Pt, res.best, st);
                count = best != kNoBest;
            }
            res.count = count;
        }
        if (MODE != RSI_MODE_BOOL && C.out.hit_idx)
            compact<MODE>(C.out, valid && count > 0, i, res, dist, Pt);
    }
}

template <int MODE, bool STATS, bool LEAFN>
__global__ void __maxnreg__(PacketRegs<MODE>::value) k_trace_packet(TraceParams P) {
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
    C.order = P.order;
    C.status = P.status;
    C.out = P.out;
    TravStats st = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
    unsigned long long segs = 0;
    if (C.coarse)
        packet_loop<MODE, STATS, LEAFN, true>(C, P.root, P.walk_work, st, segs);
    else
        packet_loop<MODE, STATS, LEAFN, false>(C, P.root, P.walk_work, st, segs);
    walk_finish(P.walk_work);
    if (STATS) flush_stats(st, P.stats, segs);
}

using PacketFn = void (*)(TraceParams);

template <bool STATS, bool LEAFN>
static PacketFn pick_packet(int mode) {
    if (mode == RSI_MODE_BOOL) return k_trace_packet<RSI_MODE_BOOL, STATS, LEAFN>;
    if (mode == RSI_MODE_COUNT) return k_trace_packet<RSI_MODE_COUNT, STATS, LEAFN>;
    return k_trace_packet<RSI_MODE_NEAREST, STATS, LEAFN>;
}

static PacketFn packet_kernel(int mode, bool stats, bool leafn) {
    if (stats) return leafn ? pick_packet<true, true>(mode) : pick_packet<true, false>(mode);
    return leafn ? pick_packet<false, true>(mode) : pick_packet<false, false>(mode);
}

cudaError_t launch_trace_packet(const TraceParams& P, int mode, bool stats, cudaStream_t s) {
    PacketFn fn = packet_kernel(mode, stats, P.leaf_size > 1);
    TraceParams Q = P;
    Q.root = walk_start(0, P.nT, P.leaf_size);
    int grid = 0;
    cudaError_t e = occupancy_grid((const void*)fn, kPacketBlock, 0, &grid);
    if (e != cudaSuccess) return e;
    const int64_t warps_needed = (P.nR + 31) / 32;
    const int64_t blocks_needed = (warps_needed + kPacketBlock / 32 - 1) / (kPacketBlock / 32);
    if (blocks_needed < grid) grid = (int)blocks_needed;
    if (grid < 1) grid = 1;
    if (P.out.hit_idx) {
        e = cudaMemsetAsync(P.out.n_hits, 0, sizeof(int64_t), s);
        if (e != cudaSuccess) return e;
    }
    fn<<<grid, kPacketBlock, 0, s>>>(Q);
    return cudaGetLastError();
}

}  // namespace rsi
