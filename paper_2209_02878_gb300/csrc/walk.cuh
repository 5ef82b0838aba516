// Traversal loop of the default path: one segment per lane, over four-way
// records of the tree (exact binary nodes where those are too coarse), all in
// global memory.  traverse_core.cuh holds the general loop that serves the
// other options: smaller stacks, 4-wide exact nodes, treelets.
//
// What bounds it is instruction issue, the divergence between lanes and L1
// wavefronts (one per 32-byte sector that a lane reads), not DRAM bytes (the
// tree sits in L1 / L2).
//
// So the loop is split into three phases that each run with many lanes at
// once (which one is next: walk_phase.h):
//  - node steps: every lane whose current item is a node tests the node's
//    four child boxes and moves on (leaf children are items like nodes:
//    entered or pushed, not tested here);
//  - triangle tests: lanes whose current item is a leaf wait until several of
//    them do (inline, the test ran for 1.2 of 32 lanes on average);
//  - refill: finished lanes write their results together and take new
//    segments that the whole warp has set up 32 at a time in shared memory.
// A phase runs when kStall lanes cannot take a node step, the one with more
// lanes waiting first.  NEAREST keeps only the best crossing's position and
// interval across the loop (its outputs are recomputed once, when written),
// which leaves it 68 B of spills at 80 registers (166 in the general loop).
//
// And a node step takes two levels of the binary tree at once, from a 64-byte
// record of the four grandchildren's boxes on a 15-bit grid over the mesh's
// box: as many bytes and boxes per segment as binary steps on 32-byte grid
// nodes, but half the steps, each of which costs a ballot, the stack and the
// loop beside its boxes, and half the chain of dependent reads.  (Exact boxes
// take twice the bytes.)  The 16-bit half that holds a face becomes a float in
// [1, 2) by one byte permutation, whose selector also chooses the near or the
// far face, so the decoding costs what that choice costs anyway.
//
// us, general loop -> this one: 10M random segments over a 29,768-triangle
// terrain boolean 1,179 -> 708, count 1,780 -> 1,021, nearest 2,202 -> 1,330,
// nearest of its raster 2,317 -> 1,386; 1M segments over a 1.31M-triangle sphere
// boolean 536 -> 283, count 1,462 -> 749, nearest 1,075 -> 601.  Boolean on the
// terrain: warp instructions 954M -> 535M, active lanes 14.4 -> 23.3.
#pragma once

#include "traverse_core.cuh"
#include "walk_phase.h"

namespace rsi {

constexpr int kDone = (int)0x80000000;  // no item: the segment is finished
// A radix tree over 62-bit keys is at most 63 deep: 32 steps of two levels that
// push at most three items each, or 63 binary ones that push one.
constexpr int kWalkStack = 96;
// Lanes without a node step that end the node phase: fewer keep the lanes
// busier, more run the other phases fuller (NEAREST has the dearest ones).
// Boolean and count at 12 / 16 / 20: 758 / 751 / - and 1,072 / 1,056 / - us on
// the 29,768-triangle terrain with 10M random segments (762 and 1,116 at 20
// with 72 registers); nearest at 16 / 20 / 24: 1,343 / 1,336 / 1,391 us there,
// 1,406 / 1,345 / 1,283 of its raster, 610 / 604 / 616 of the sphere.
template <int MODE>
constexpr int kStall = MODE == RSI_MODE_NEAREST ? 20 : 16;

// Whether a lane keeps its segment's end points and index, which node steps do
// not need, in shared memory instead of seven registers, and the registers of
// the kernels.  BOOL then fits 72 without a spill and COUNT with 4 B (28 warps
// per SM): boolean on the terrain above 697 us, 744 at 80 registers without;
// count 994 and 1,061.  NEAREST, which also needs them for its outputs, does
// not gain: nearest of the raster 1,365 us with at its best, 1,345 without.
template <int MODE>
constexpr bool kOwn = MODE != RSI_MODE_NEAREST;
template <int MODE>
constexpr int kWalkRegs = MODE == RSI_MODE_NEAREST ? 80 : 72;
// The batch's kernels hold an item's pointers as well, and run side by side: 80 /
// 96 / 112 / 128: 1,215 / 1,143 / 1,180 / 1,151 us on 16 meshes with 3.5M
// segments; with the end points of boolean segments in shared memory 1,173.
constexpr int kBatchRegs = 96;

// Byte selectors that turn the low / high half of a node word into a float.
constexpr unsigned kSelLo = 0x7104u, kSelHi = 0x7324u, kSelFar = kSelLo ^ kSelHi;

// The nodes' grid has 32,760 steps across the mesh; where that is too coarse for
// its detail (rsi_internal.cuh) the loop reads the exact binary nodes.
__device__ __forceinline__ bool walk_coarse(int2 coarse, int n) {
    return coarse.x > n / 8 || coarse.y > kBlurredLeaves;
}

// A lane's segment: end points for the triangle test and, per axis, the
// constants of the box test in the grid's coordinates
//   entry parameter = fma(near face, i, n),  exit = fma(far face, i, f),
// and the byte selectors that take the near / far face out of a node word.
struct WalkSeg {
    float ax_, ay_, az_, dx, dy, dz;
    float ix, iy, iz, nx, ny, nz, fx, fy, fz;
    unsigned swap;        // 32 on odd lanes (walk_node4)
    unsigned ex, ey, ez;  // selectors of the near faces (far: ^ kSelFar)
    float md;
    bool fp64only;
    __device__ __forceinline__ void select() {
        // held as values: recomputed at every node they cost nine instructions
        ex = ix < 0.f ? kSelHi : kSelLo;
        ey = iy < 0.f ? kSelHi : kSelLo;
        ez = iz < 0.f ? kSelHi : kSelLo;
        swap = (threadIdx.x & 1) * 32u;
        asm volatile("" : "+r"(ex), "+r"(ey), "+r"(ez));
    }
    __device__ __forceinline__ float ax() const { return ax_; }
    __device__ __forceinline__ float ay() const { return ay_; }
    __device__ __forceinline__ float az() const { return az_; }
    __device__ __forceinline__ void range() {  // the triangle test's scale of d
        md = maxabs3(dx, dy, dz);
        fp64only = !(md >= kRangeLo && md <= kRangeHi);
    }
};

// Box-test constants of one axis (u = 2^-24) for the segment coordinates
// X(a) = base + (a - o) s and D = d s, with base = 1 on the grid and o = 0,
// s = 1, base = 0 (exact) for the exact nodes; d = fl(b - a).
// i = rcp.approx(D) (1 ulp) is (1 / D_exact)(1 + e), |e| <= 5u (d, D and the
// reciprocal), and X(a) is off by at most 3u |X(a)| + 2u, or exact (s = 1).
// c = fl(X(a) i); a face at X has the exact parameter (X - X_exact(a)) / D_exact,
// and X i - c is that times (1 + e), up to 4u |c| + 2u |i| (exact nodes: u |c|).
// The constants are n = -(c + pad) and f = pad - c with pad = 8u |c| + 4u |i| +
// 16u: the first two terms cover those errors and the rounding of n / f (u |c|),
// and 16u the relative errors e and the fma's own rounding for every parameter
// in [0, 1].  The exact nodes go without 4u |i|: in their coordinates it would
// move every face by 2.4e-7 whatever the mesh's size (segments 1e-5 long: 16
// triangle tests each instead of 1.5; 2e-7 long: every triangle).  So for a box
// that the exact segment meets at parameters [s0, s1] within [0, 1], the
// computed entry is below s0 and the computed exit above s1, strictly, and
// stays so after both are clamped to [0, 1]: `entry < exit` never rejects it.
//  - |D| < 2^-62 (a zero component, and every tiny one): i = 2^62, pad = 2 +
//    8u |c| + 4u i (grid).  A segment inside the slab gets entry <= 0 and exit >= 1.
//  - |D| > 2^100 (or infinite) or |c| > 2^100: i = 0, n = -2, f = 2: the
//    axis never rejects.
// Empty boxes: in the exact nodes both faces are +inf, which is always rejected
// (entry = exit after the clamp; NaN clamps to 0).  On the grid lo is far beyond
// hi, and what a segment of a million mesh sizes enters all the same is the
// null triangle, or triangles without valid vertices: never hit.
__device__ __forceinline__ void walk_axis(float a, float d, float o, float s, float base, float& i,
                                          float& n, float& f) {
    const float X = __fmaf_rn(__fsub_rn(a, o), s, base), D = __fmul_rn(d, s);
    const float ad = fabsf(D);
    const bool flat = ad < 0x1p-62f;
    i = flat ? 0x1p62f : rcp_approx(D);
    const float c = __fmul_rn(X, i);
    const float pad = __fmaf_rn(fabsf(c), 0x1p-21f,
                                __fmaf_rn(fabsf(i), base * 0x1p-22f, flat ? 2.f : 0x1p-20f));
    n = -__fadd_rn(c, pad);
    f = __fsub_rn(pad, c);
    if (!(ad <= 0x1p100f && fabsf(c) <= 0x1p100f)) {
        i = 0.f;
        n = -2.f;
        f = 2.f;
    }
}

// A grid coordinate of a node word as a float: the chosen 16 bits (bit 15 set)
// become bits 8..23 under 0x3f: 1 + q 2^-15.
__device__ __forceinline__ float grid_face(unsigned w, unsigned sel) {
    return __uint_as_float(__byte_perm(w, 0x3f000000u, sel));
}

// Half a grid record in one 256-bit read-only load.
__device__ __forceinline__ void ld_qnode(const float4* p, unsigned w[8]) {
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]),
          "=r"(w[7])
        : "l"(p));
}

__device__ __forceinline__ float fma_sat(float a, float b, float c) {
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Entry parameter of a box with the given near and far faces (clamped to
// [0, 1]) and whether the segment's part [0, tlim] may meet it.  The clamps
// come with the fma, so an axis costs two of them and the choice of faces.
template <bool LIMIT>
__device__ __forceinline__ bool walk_box(const WalkSeg& s, float ex, float ey, float ez, float gx,
                                         float gy, float gz, float tlim, float& tn) {
    tn = max3(fma_sat(ex, s.ix, s.nx), fma_sat(ey, s.iy, s.ny), fma_sat(ez, s.iz, s.nz));
    float tf = min3(fma_sat(gx, s.ix, s.fx), fma_sat(gy, s.iy, s.fy), fma_sat(gz, s.iz, s.fz));
    if (LIMIT) tf = fminf(tf, tlim);
    return tn < tf;
}

// Leaf items: ~position of a one-triangle leaf, or, with LEAFN (leaf sizes
// above 1), ~(8 position + count - 1).
template <bool LEAFN>
__device__ __forceinline__ int walk_item(int ref, int cnt) {
    return cnt > 0 ? ~(LEAFN ? ref << 3 | (cnt - 1) : ref) : ref;
}

// A node's children: whether the segment enters each, entry parameters and
// items.  The two children of the exact binary node:
template <bool LIMIT, bool LEAFN>
__device__ __forceinline__ void walk_node2(const TraceCtx& C, const WalkSeg& s, int node, float tlim,
                                           bool h[2], float t[2], int x[2]) {
    ulonglong2 q0, q1, q2;
    int4 rc;
    ld_node(C.nodes + 4 * (int64_t)node, q0, q1, q2, rc);
    const float2 lx = up2(q0.x), ly = up2(q0.y), lz = up2(q1.x);
    const float2 hx = up2(q1.y), hy = up2(q2.x), hz = up2(q2.y);
    const bool gx = s.ix < 0.f, gy = s.iy < 0.f, gz = s.iz < 0.f;
    h[0] = walk_box<LIMIT>(s, gx ? hx.x : lx.x, gy ? hy.x : ly.x, gz ? hz.x : lz.x,
                           gx ? lx.x : hx.x, gy ? ly.x : hy.x, gz ? lz.x : hz.x, tlim, t[0]);
    h[1] = walk_box<LIMIT>(s, gx ? hx.y : lx.y, gy ? hy.y : ly.y, gz ? hz.y : lz.y,
                           gx ? lx.y : hx.y, gy ? ly.y : hy.y, gz ? lz.y : hz.y, tlim, t[1]);
    x[0] = walk_item<LEAFN>(rc.x, rc.z);
    x[1] = walk_item<LEAFN>(rc.y, rc.w);
}

// The four children of a 64-byte grid record.  Odd lanes read the halves in
// the other order (it does not matter which is which): a record's first
// halves all lie in two of L1's four 32-byte bank groups.
template <bool LIMIT>
__device__ __forceinline__ void walk_node4(const TraceCtx& C, const WalkSeg& s, int node, float tlim,
                                           bool h[4], float t[4], int x[4]) {
    const float4* p = C.qnodes + 4 * (int64_t)node;
    unsigned w[16];
    ld_qnode((const float4*)((uintptr_t)p ^ s.swap), w);
    ld_qnode((const float4*)((uintptr_t)p ^ s.swap ^ 32u), w + 8);
    const unsigned gx = s.ex ^ kSelFar, gy = s.ey ^ kSelFar, gz = s.ez ^ kSelFar;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned* c = w + 8 * (k >> 1) + 3 * (k & 1);
        h[k] = walk_box<LIMIT>(s, grid_face(c[0], s.ex), grid_face(c[1], s.ey),
                               grid_face(c[2], s.ez), grid_face(c[0], gx), grid_face(c[1], gy),
                               grid_face(c[2], gz), tlim, t[k]);
        x[k] = (int)w[8 * (k >> 1) + 6 + (k & 1)];
    }
}

// End points and box-test constants of segment i (not md and fp64only);
// returns whether its coordinates are finite.
__device__ __forceinline__ bool walk_setup(const TraceCtx& C, int64_t i, WalkSeg& w) {
    w.ax_ = C.A[3 * i];
    w.ay_ = C.A[3 * i + 1];
    w.az_ = C.A[3 * i + 2];
    const float bx = C.B[3 * i], by = C.B[3 * i + 1], bz = C.B[3 * i + 2];
    w.dx = __fsub_rn(bx, w.ax_);
    w.dy = __fsub_rn(by, w.ay_);
    w.dz = __fsub_rn(bz, w.az_);
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 g = make_float4(1.f, 1.f, 1.f, 0.f);
    if (!C.coarse && C.frame) {
        o = ld4(C.frame);
        g = ld4(C.frame + 1);
    }
    const float base = C.coarse ? 0.f : 1.f;
    walk_axis(w.ax_, w.dx, o.x, g.x, base, w.ix, w.nx, w.fx);
    walk_axis(w.ay_, w.dy, o.y, g.y, base, w.iy, w.ny, w.fy);
    walk_axis(w.az_, w.dz, o.z, g.z, base, w.iz, w.nz, w.fz);
    return finite3(w.ax_, w.ay_, w.az_) && finite3(bx, by, bz);
}

// Segments set up by a warp and not yet taken by a lane (shared memory, one
// per warp): four 16-byte words per segment.
// And, with OWN, each lane's own segment {a, index}, {d, -}.
template <bool OWN>
struct WalkStage {
    float4 q[4][32];
    float4 own[OWN ? 2 : 1][OWN ? 32 : 1];
};

// Best crossing of a NEAREST segment: leaf position (kBest64: decided in
// FP64), and the interval that holds its t.  Everything else about it is
// recomputed once, when the result is written.
constexpr unsigned kNoBest = 0xffffffffu, kBest64 = 0x80000000u;

// Test segment i against the triangles of leaf `item`; s.range() is up to
// date.  Returns true when BOOL found a crossing.
template <int MODE, bool STATS, bool LEAFN>
__device__ __forceinline__ bool walk_leaf(const TraceCtx& C, const WalkSeg& s, int64_t i, int item,
                                          int& count, unsigned& best, float& tlo, float& tlim,
                                          TravStats& st) {
    const int pos0 = LEAFN ? (int)((unsigned)~item >> 3) : ~item;
    const int pos1 = LEAFN ? pos0 + (~item & 7) : pos0;
    for (int pos = pos0; pos <= pos1; ++pos) {
        const float4* tp = C.tris + 3 * (int64_t)pos;
        const float4 a = ld4(tp), b = ld4(tp + 1), c = ld4(tp + 2);
        float t = 0.f, u = 0.f, v = 0.f, err = 0.f;
        if (STATS) ++st.tests;
        int r = mt32(s, a, b, c, MODE == RSI_MODE_NEAREST, t, u, v, err);
        unsigned code = (unsigned)pos;
        if (r == 2) {
            if (STATS) ++st.fp64;
            const float* pa = C.A + 3 * i;
            const float* pb = C.B + 3 * i;
            double tuv[3];
            r = mt64(pa[0], pa[1], pa[2], pb[0], pb[1], pb[2], a, b, c,
                     MODE == RSI_MODE_NEAREST ? tuv : nullptr);
            if (MODE == RSI_MODE_NEAREST && r) {
                t = (float)tuv[0];
                err = 0x1p-23f;
                code |= kBest64;
            }
        }
        if (!r) continue;
        if (MODE == RSI_MODE_BOOL) {
            count = 1;
            return true;
        }
        if (MODE == RSI_MODE_COUNT) ++count;
        if (MODE == RSI_MODE_NEAREST) {
            bool take = best == kNoBest || t + err < tlo;
            if (!take && !(t - err > tlim)) {
                // the intervals overlap: compare the definition's t in FP64,
                // ties to the lower triangle index
                const int bpos = (int)(best & ~kBest64);
                const double tn = exact_t(C.A, C.B, i, C.tris, pos);
                const double tb = exact_t(C.A, C.B, i, C.tris, bpos);
                take = tn < tb ||
                       (tn == tb && f2i(a.w) < f2i(ld4(C.tris + 3 * (int64_t)bpos).w));
            }
            if (take) {
                best = code;
                tlo = t - err;
                tlim = fminf(1.f, t + err);
            }
        }
    }
    return false;
}

// Outputs of a NEAREST segment with best crossing `best`.
template <bool STATS>
__device__ __forceinline__ void walk_nearest_out(const TraceCtx& C, const WalkSeg& s, int64_t i,
                                                 unsigned best, float& dist, float P[3],
                                                 int& tri, TravStats& st) {
    float t = 0.f, u = 0.f, v = 0.f;
    dist = 0.f;
    P[0] = P[1] = P[2] = 0.f;
    tri = -1;
    if (best != kNoBest) {
        const float4* tp = C.tris + 3 * (int64_t)(best & ~kBest64);
        tri = f2i(ld4(tp).w);
        // the thresholds and their derivation: nearest_values
        const float dd = fmaf(s.dx, s.dx, fmaf(s.dy, s.dy, s.dz * s.dz));
        const float dlen = sqrtf(dd) * 1.0001f;
        const float thresh = 0.95f * ((1e-5f - 0x1p-24f) / fmaxf(1.f, dlen) - 0x1p-24f);
        bool exact = (best & kBest64) != 0u || s.fp64only, refine = false;
        if (!exact) {
            float euv;
            const float et = mt32_tight(s, ld4(tp), ld4(tp + 1), ld4(tp + 2), t, u, v, euv);
            refine = !(et <= thresh && euv <= 0.95e-5f);
            exact = refine && (!(et < INFINITY && dlen * et <= 4.f && euv <= 4.f) || dlen >= 64.f);
        }
        if (exact) {
            if (STATS) ++st.exact;
            float o[7];
            values64(C.A, C.B, i, ld4(tp), ld4(tp + 1), ld4(tp + 2), o);
            t = o[0];
            u = o[1];
            v = o[2];
            P[0] = o[3];
            P[1] = o[4];
            P[2] = o[5];
            dist = o[6];
        } else {
            if (refine) {
                if (STATS) ++st.refines;
                const float a3[3] = {s.ax(), s.ay(), s.az()};
                const float b3[3] = {C.B[3 * i], C.B[3 * i + 1], C.B[3 * i + 2]};
                float tuv[3];
                values_df(a3, b3, ld4(tp), ld4(tp + 1), ld4(tp + 2), tuv);
                t = tuv[0];
                u = tuv[1];
                v = tuv[2];
            }
            P[0] = fmaf(t, s.dx, s.ax());
            P[1] = fmaf(t, s.dy, s.ay());
            P[2] = fmaf(t, s.dz, s.az());
            dist = t * sqrtf(dd);
        }
    }
    const TravOut& o = C.out;
    o.tri[i] = tri;
    if (o.tuv) {
        o.tuv[3 * i] = t;
        o.tuv[3 * i + 1] = u;
        o.tuv[3 * i + 2] = v;
    }
    if (o.point) {
        o.point[3 * i] = P[0];
        o.point[3 * i + 1] = P[1];
        o.point[3 * i + 2] = P[2];
    }
    if (o.dist) o.dist[i] = dist;
}

// The stack index is clamped, so that a corrupt tree cannot leave the array;
// the step bound (walk_more) ends its walk.
__device__ __forceinline__ void walk_push(int* stack, int& sp, int x) {
    sp = min(sp + 1, kWalkStack);
    stack[sp] = x;
}

// Node steps of a warp until at most `floor_` lanes have one; returns the
// lanes that do.  The step has no branches but predicated pushes and a pop: a
// lane goes on with one of the children that it enters and pushes the others.
// NEAREST orders them, each pair by entry and the pairs by their first entry
// (as two binary steps would).
template <int MODE, bool STATS, bool LEAFN, bool COARSE>
__device__ __forceinline__ unsigned walk_steps(const TraceCtx& C, const WalkSeg& s, int& cur,
                                               int& sp, int* stack, float tlim, unsigned& left,
                                               int floor_, TravStats& st) {
    constexpr bool LIMIT = MODE == RSI_MODE_NEAREST;
    unsigned inner;
    do {
        if (cur >= 0) {
            if (STATS) ++st.visits;
            bool h[4];
            float t[4];
            int x[4];
            bool any;
            if (COARSE) {
                walk_node2<LIMIT, LEAFN>(C, s, cur, tlim, h, t, x);
                const bool first0 = h[0] && (!h[1] || t[0] <= t[1]);
                any = h[0] || h[1];
                if (h[0] && h[1]) walk_push(stack, sp, first0 ? x[1] : x[0]);
                cur = first0 ? x[0] : x[1];
            } else {
                walk_node4<LIMIT>(C, s, cur, tlim, h, t, x);
                any = h[0] || h[1] || h[2] || h[3];
                if (LIMIT) {
                    const bool a = h[0] && (!h[1] || t[0] <= t[1]);
                    const bool b = h[2] && (!h[3] || t[2] <= t[3]);
                    const bool anya = h[0] || h[1], anyb = h[2] || h[3];
                    const bool two_a = h[0] && h[1], two_b = h[2] && h[3];
                    const bool f = anya && (!anyb || (a ? t[0] : t[1]) <= (b ? t[2] : t[3]));
                    const int na = a ? x[0] : x[1], fa = a ? x[1] : x[0];
                    const int nb = b ? x[2] : x[3], fb = b ? x[3] : x[2];
                    if (f ? two_b : two_a) walk_push(stack, sp, f ? fb : fa);
                    if (anya && anyb) walk_push(stack, sp, f ? nb : na);
                    if (f ? two_a : two_b) walk_push(stack, sp, f ? fa : fb);
                    cur = f ? na : nb;
                } else {
                    cur = x[0];
                    if (h[1]) {
                        if (h[0]) walk_push(stack, sp, cur);
                        cur = x[1];
                    }
                    if (h[2]) {
                        if (h[0] || h[1]) walk_push(stack, sp, cur);
                        cur = x[2];
                    }
                    if (h[3]) {
                        if (h[0] || h[1] || h[2]) walk_push(stack, sp, cur);
                        cur = x[3];
                    }
                }
            }
            if (!any) cur = stack[sp--];
        }
        inner = __ballot_sync(0xffffffffu, cur >= 0);
    } while (walk_more(left, __popc(inner), floor_));
    return inner;
}

// Persistent per-warp loop over the segments [pool, pool_end) and, while `more`,
// those that next(pool, pool_end) fetches (it returns false when there are
// none; warp-uniform); order, streamed input and compaction as in trace_loop.
// Segment indices fit 31 bits (walk_fits).  `start` is the first item of every
// segment: the Karras root's slot, the whole mesh as one leaf, or kNoRoot.
// Must be called by all 32 lanes of the warp; sg is the warp's own.
template <int MODE, bool STATS, bool LEAFN, bool OWN, typename Next>
__device__ __forceinline__ void walk_loop(const TraceCtx& C, WalkStage<OWN>& sg, int start,
                                          unsigned pool, unsigned pool_end, bool more,
                                          const Next& next, TravStats& st,
                                          unsigned long long& segs) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int head = 0, avail = 0;         // staged segments not yet taken
    int cur = kDone, sp = 0;
    int count = 0;                   // BOOL / COUNT: crossings
    unsigned best = kNoBest;         // NEAREST
    float tlo = 0.f, tlim = 1.f;     // NEAREST: bounds of the best crossing's t
    WalkSeg s;
    int i = -1;                      // this lane's segment (-1: none)
    if (OWN) sg.own[0][lane].w = i2f(-1);
    int stack[kWalkStack + 1];
    stack[0] = kDone;
    unsigned left = walk_bound(C.max_visits);  // node steps until the next refill
    unsigned inner = 0u;  // lanes with a node step
    while (true) {
        const unsigned dead = __ballot_sync(FULL, cur == kDone);
        const unsigned leaf = ~(inner | dead);
        const bool refillable = avail > 0 || pool < pool_end || more;
        const int nd = __popc(dead), nl = __popc(leaf);
        const WalkPhase phase = walk_phase(nd, nl, refillable, kStall<MODE>);
        if (phase == kPhaseRefill) {
            // ---- refill: results of the finished segments, then new ones
            left = walk_bound(C.max_visits);
            float dist = 0.f, P[3] = {0.f, 0.f, 0.f};
            Result res;
            if (OWN) i = f2i(sg.own[0][lane].w);
            const bool fin = cur == kDone && i >= 0;
            if (fin) {
                if (MODE == RSI_MODE_BOOL) {
                    C.out.flag[i] = (uint8_t)(count > 0);
                } else if (MODE == RSI_MODE_COUNT) {
                    C.out.count[i] = count;
                } else {
                    s.range();
                    walk_nearest_out<STATS>(C, s, i, best, dist, P, res.best, st);
                    count = best != kNoBest;
                }
                res.count = count;
            }
            if (MODE != RSI_MODE_BOOL && C.out.hit_idx)
                compact<MODE>(C.out, fin && count > 0, i, res, dist, P);
            if (fin) {
                i = -1;
                if (OWN) sg.own[0][lane].w = i2f(-1);
            }
            if (!refillable) break;  // every lane is finished
            unsigned idle = dead;
            while (true) {
                if (avail == 0) {  // set up the next segments, one per lane
                    if (pool >= pool_end) {
                        more = more && next(pool, pool_end);
                        if (!more) break;
                    }
                    const int take = (int)min(pool_end - pool, 32u);
                    bool ok = false;
                    WalkSeg w;
                    unsigned k = 0u;
                    if (lane < take) {
                        int64_t kk = (int64_t)pool + lane;
                        bool known = true;
                        if (C.order) {  // a caller's order: entries outside [0, nR) are skipped
                            kk = C.order[kk];
                            known = kk >= 0 && kk < C.nR;
                            if (!known) atomicCAS(C.status, 0, RSI_ERR_BAD_INDEX);
                        }
                        if (STATS) ++segs;
                        if (known) {
                            k = (unsigned)kk;
                            ok = walk_setup(C, kk, w) && start != kNoRoot;
                            if (!ok) {  // non-finite segment or empty mesh: a miss
                                float q0, q1[3];
                                int tri;
                                if (MODE == RSI_MODE_BOOL)
                                    C.out.flag[kk] = 0;
                                else if (MODE == RSI_MODE_COUNT)
                                    C.out.count[kk] = 0;
                                else
                                    walk_nearest_out<STATS>(C, w, kk, kNoBest, q0, q1, tri, st);
                            }
                        }
                    }
                    const unsigned good = __ballot_sync(FULL, ok);
                    __syncwarp();  // the entries before these have been read
                    if (ok) {
                        const int e = __popc(good & lt);
                        sg.q[0][e] = make_float4(w.ax_, w.ay_, w.az_, i2f((int)k));
                        sg.q[1][e] = make_float4(w.dx, w.dy, w.dz, w.fz);
                        sg.q[2][e] = make_float4(w.ix, w.iy, w.iz, w.nx);
                        sg.q[3][e] = make_float4(w.ny, w.nz, w.fx, w.fy);
                    }
                    __syncwarp();
                    pool += take;
                    head = 0;
                    avail = __popc(good);
                    if (avail == 0) continue;
                }
                const int want = __popc(idle), n = min(avail, want);
                const int r = __popc(idle & lt);
                if (cur == kDone && r < n) {
                    const float4 q0 = sg.q[0][head + r], q1 = sg.q[1][head + r];
                    const float4 q2 = sg.q[2][head + r], q3 = sg.q[3][head + r];
                    if (OWN) {
                        sg.own[0][lane] = q0;
                        sg.own[1][lane] = q1;
                    } else {
                        s.ax_ = q0.x;
                        s.ay_ = q0.y;
                        s.az_ = q0.z;
                        s.dx = q1.x;
                        s.dy = q1.y;
                        s.dz = q1.z;
                        i = f2i(q0.w);
                    }
                    s.fz = q1.w;
                    s.ix = q2.x;
                    s.iy = q2.y;
                    s.iz = q2.z;
                    s.nx = q2.w;
                    s.ny = q3.x;
                    s.nz = q3.y;
                    s.fx = q3.z;
                    s.fy = q3.w;
                    s.select();
                    cur = start;
                    sp = 0;
                    count = 0;
                    best = kNoBest;
                    tlim = 1.f;
                }
                head += n;
                avail -= n;
                if (n == want) break;
                idle = __ballot_sync(FULL, cur == kDone);
            }
            inner = __ballot_sync(FULL, cur >= 0);
            continue;
        }
        if (phase == kPhaseLeaves) {
            // ---- triangle tests of the waiting leaves
            if (cur < 0 && cur != kDone) {
                if (OWN) {  // the end points, for this phase only
                    const float4 a = sg.own[0][lane], d = sg.own[1][lane];
                    s.ax_ = a.x;
                    s.ay_ = a.y;
                    s.az_ = a.z;
                    s.dx = d.x;
                    s.dy = d.y;
                    s.dz = d.z;
                    i = f2i(a.w);
                }
                s.range();
                const bool stop = walk_leaf<MODE, STATS, LEAFN>(C, s, i, cur, count, best, tlo,
                                                                tlim, st);
                cur = MODE == RSI_MODE_BOOL && stop ? kDone : stack[sp--];
            }
            inner = __ballot_sync(FULL, cur >= 0);
            continue;
        }
        // ---- node steps until kStall lanes (a quarter of those left at the
        // end of the work) have none
        const int floor_ = walk_floor(nd, refillable, kStall<MODE>);
        inner = C.coarse ? walk_steps<MODE, STATS, LEAFN, true>(C, s, cur, sp, stack, tlim, left,
                                                                floor_, st)
                         : walk_steps<MODE, STATS, LEAFN, false>(C, s, cur, sp, stack, tlim, left,
                                                                 floor_, st);
        if (left == 0u) {
            if (lane == 0) atomicCAS(C.status, 0, RSI_ERR_INTERNAL);
            cur = kDone;
            inner = 0u;
        }
    }
}

// Source of segments of a launch over one mesh: chunks of C.fetch from a
// counter.
struct WalkCounter {
    const TraceCtx& C;
    unsigned long long* counter;
    __device__ __forceinline__ bool operator()(unsigned& pool, unsigned& pool_end) const {
        unsigned long long b = 0ull;
        if ((threadIdx.x & 31) == 0) b = atomicAdd(counter, (unsigned long long)C.fetch);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b >= (unsigned long long)C.nR) return false;
        pool = (unsigned)b;
        pool_end = (unsigned)min((long long)(b + C.fetch), (long long)C.nR);
        // streamed input: see trace_loop
        if (C.ready && !wait_flag(C.ready + (int64_t)(pool_end - 1) / C.ready_chunk, C.status,
                                  C.wait_polls)) {
            if ((threadIdx.x & 31) == 0) atomicMax(counter, (unsigned long long)C.nR);
            pool = pool_end;
            return false;
        }
        return true;
    }
};

struct WalkNone {
    __device__ __forceinline__ bool operator()(unsigned&, unsigned&) const { return false; }
};

// End of a block of a launch whose warps took work from counter[0]: the last
// block clears it and the count of finished blocks (counter[1]) for the next
// launch.  A memset before each launch cost as much as a tenth of the
// smallest queries.  All threads of the block call it.
__device__ __forceinline__ void walk_finish(unsigned long long* counter) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(counter + 1, 1ull) == (unsigned long long)gridDim.x - 1ull) {
            counter[0] = 0ull;
            counter[1] = 0ull;
        }
    }
}

}  // namespace rsi
