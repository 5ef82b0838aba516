// Traversal loop of the default path: one segment per lane, binary nodes,
// the whole tree in global memory (no treelet copy), a 64-entry stack.
// traverse_core.cuh holds the general loop that serves the other options.
//
// What bounds it is instruction issue, the divergence between lanes and L1
// wavefronts (one per 32-byte sector that a lane reads), not DRAM bytes (the
// tree sits in L1 / L2).  So the loop is split into three phases that each run
// with many lanes at once:
//  - node steps: every lane whose current item is a node tests the node's two
//    child boxes and moves on (leaf children are items like nodes: entered
//    or pushed, not tested here);
//  - triangle tests: lanes whose current item is a leaf wait until several of
//    them do (inline, the test ran for 1.2 of 32 lanes on average);
//  - refill: finished lanes write their results together and take new
//    segments that the whole warp has set up 32 at a time in shared memory.
// A phase runs when kStall lanes cannot take a node step, the one with more
// lanes waiting first.  Against one loop that does all three for each lane
// where it stands: 954M -> 610M warp instructions and 14.4 -> 22.9 active
// lanes on the paper-scale boolean query; boolean 1,177 -> 1,010 us, nearest
// 2,212 -> 1,615 us there, nearest of the raster 2,291 -> 1,498 us, of the
// 131,072-triangle terrain with 262,144 segments 238 -> 147 us, of the
// 1.31M-triangle sphere with 1M segments 1,100 -> 796 us.  NEAREST keeps only
// the best crossing's position and interval across the loop (its outputs are
// recomputed once, when written), which takes its spills away.
#pragma once

#include "traverse_core.cuh"

namespace rsi {

constexpr int kDone = (int)0x80000000;  // no item: the segment is finished
constexpr int kWalkStack = 64;          // a radix tree over 62-bit keys is at most 63 deep
// Lanes without a node step that end the node phase.  12 / 16 / 20 (72
// registers): boolean 1,014 / 1,010 / 1,045 us on the 29,768-triangle terrain
// with 10M random segments, nearest 1,563 / 1,498 / - us under its raster.
constexpr int kStall = 16;

// 72 registers (28 warps per SM): at 64 the loop spills (boolean 1,069 against
// 1,010 us, count 1,562 against 1,386), at 80 fewer warps hide less (1,034,
// 1,459); nearest 1,615 us at 72, 1,604 at 64, 1,656 at 80.
constexpr int kWalkRegs = 72;

// A lane's segment: end points for the triangle test and, per axis, the
// constants of the box test
//   entry parameter = fma(near face, i, n),  exit = fma(far face, i, f).
struct WalkSeg {
    float ax_, ay_, az_, dx, dy, dz;
    float ix, iy, iz, nx, ny, nz, fx, fy, fz;
    float md;
    bool fp64only;
    __device__ __forceinline__ float ax() const { return ax_; }
    __device__ __forceinline__ float ay() const { return ay_; }
    __device__ __forceinline__ float az() const { return az_; }
    __device__ __forceinline__ void range() {  // the triangle test's scale of d
        md = maxabs3(dx, dy, dz);
        fp64only = !(md >= kRangeLo && md <= kRangeHi);
    }
};

// Box-test constants of one axis (u = 2^-24).  With d = fl(b - a) (relative
// error u) and i = rcp.approx(d) (1 ulp), i = (1 / d_exact)(1 + e), |e| <= 4u.
// c = fl(a i); a face at x has the exact parameter s = (x - a) / d_exact and
// x i - c = s (1 + e) + at most u |c|.  The constants are n = -(c + pad) and
// f = pad - c with pad = 4u |c| + 16u: 4u |c| covers the roundings of c and of
// n / f, and 16u the relative errors e and the fma's own rounding for every
// parameter in [0, 1].  So for a box that the exact segment meets at
// parameters [s0, s1] within [0, 1], the computed entry is below s0 and the
// computed exit above s1, strictly, and stays so after both are clamped to
// [0, 1]: `entry < exit` never rejects it.
//  - |d| < 2^-62 (a zero component, and every tiny one): i = 2^62, pad = 2 +
//    4u |c|.  A segment inside the slab gets entry <= 0 and exit >= 1; one
//    that is outside by more than about 2^-61 + 4u |a| is rejected.
//  - |d| > 2^100 (or infinite) or |c| > 2^100: i = 0, n = -2, f = 2: the
//    axis never rejects.
// Empty boxes (both faces +inf) give entry = exit after the clamp (NaN clamps
// to 0): always rejected.
__device__ __forceinline__ void walk_axis(float a, float d, float& i, float& n, float& f) {
    const float ad = fabsf(d);
    const bool flat = ad < 0x1p-62f;
    i = flat ? 0x1p62f : rcp_approx(d);
    const float c = __fmul_rn(a, i);
    const float pad = __fmaf_rn(fabsf(c), 0x1p-22f, flat ? 2.f : 0x1p-20f);
    n = -__fadd_rn(c, pad);
    f = __fsub_rn(pad, c);
    if (!(ad <= 0x1p100f && fabsf(c) <= 0x1p100f)) {
        i = 0.f;
        n = -2.f;
        f = 2.f;
    }
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

// Entry parameter of the box (clamped to [0, 1]) and whether the segment's
// part [0, tlim] may meet it.  The clamps come with the fma, so an axis costs
// two of them and the selection of the near face.
template <bool LIMIT>
__device__ __forceinline__ bool walk_box(const WalkSeg& s, float lx, float ly, float lz, float hx,
                                         float hy, float hz, float tlim, float& tn) {
    const bool gx = s.ix < 0.f, gy = s.iy < 0.f, gz = s.iz < 0.f;
    tn = max3(fma_sat(gx ? hx : lx, s.ix, s.nx), fma_sat(gy ? hy : ly, s.iy, s.ny),
              fma_sat(gz ? hz : lz, s.iz, s.nz));
    float tf = min3(fma_sat(gx ? lx : hx, s.ix, s.fx), fma_sat(gy ? ly : hy, s.iy, s.fy),
                    fma_sat(gz ? lz : hz, s.iz, s.fz));
    if (LIMIT) tf = fminf(tf, tlim);
    return tn < tf;
}

// Segments set up by a warp and not yet taken by a lane (shared memory, one
// per warp): four 16-byte words per segment.
struct WalkStage {
    float4 q[4][32];
};

// Leaf items: ~position of a one-triangle leaf, or, with LEAFN (leaf sizes
// above 1), ~(8 position + count - 1).
template <bool LEAFN>
__device__ __forceinline__ int walk_item(int ref, int cnt) {
    if (!LEAFN) return ref;
    return cnt > 0 ? ~((~ref << 3) | (cnt - 1)) : ref;
}

// Best crossing of a NEAREST segment: leaf position (kBest64: decided in
// FP64), and the interval that holds its t.  Everything else about it is
// recomputed once, when the result is written.
constexpr unsigned kNoBest = 0xffffffffu, kBest64 = 0x80000000u;

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
        Result r;
        result_init(r);
        r.best = tri;
        r.bpos = (int)(best & ~kBest64);
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

// Persistent per-warp loop over segments [lo, hi) (work distribution, order,
// streamed input and compaction as trace_loop).  `start` is the first item
// of every segment: the Karras root's slot, the whole mesh as one leaf, or
// kNoRoot.  Must be called by all 32 lanes of the warp; sg is the warp's own.
template <int MODE, bool STATS, bool LEAFN>
__device__ __forceinline__ void walk_loop(const TraceCtx& C, WalkStage& sg, int start,
                                          unsigned long long* counter, int64_t lo, int64_t hi,
                                          TravStats& st, unsigned long long& segs) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int64_t pool = lo, pool_end = counter ? lo : hi;
    bool more = counter != nullptr;  // the counter may hold more chunks
    int head = 0, avail = 0;         // staged segments not yet taken
    unsigned i = kNoBest;            // this lane's segment (kNoBest: none)
    int cur = kDone, sp = 0;
    int count = 0;                   // BOOL / COUNT: crossings
    unsigned best = kNoBest;         // NEAREST
    float tlo = 0.f, tlim = 1.f;     // NEAREST: bounds of the best crossing's t
    WalkSeg s;
    int stack[kWalkStack + 1];
    stack[0] = kDone;
    // node steps between two refills: each of the 32 segments takes at most
    // max_visits, so more can only be a corrupt tree
    unsigned steps = 0;
    const unsigned bound =
        (unsigned)C.max_visits < 1u << 26 ? 32u * (unsigned)C.max_visits + 64u : 0xffffffffu;
    while (true) {
        const unsigned dead = __ballot_sync(FULL, cur == kDone);
        const unsigned leaf = __ballot_sync(FULL, cur < 0) & ~dead;
        const bool refillable = avail > 0 || pool < pool_end || more;
        const int nd = __popc(dead), nl = __popc(leaf);
        if (dead == FULL || (refillable && nd >= nl && nd + nl >= kStall)) {
            // ---- refill: results of the finished segments, then new ones
            steps = 0;
            float dist = 0.f, P[3] = {0.f, 0.f, 0.f};
            Result res;
            const bool fin = cur == kDone && i != kNoBest;
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
            if (fin) i = kNoBest;
            if (!refillable) break;  // every lane is finished
            unsigned idle = dead;
            while (idle) {
                if (avail == 0) {  // set up the next segments, one per lane
                    if (pool >= pool_end) {
                        if (!more) break;
                        unsigned long long b = 0ull;
                        if (lane == 0) b = atomicAdd(counter, (unsigned long long)C.fetch);
                        b = __shfl_sync(FULL, b, 0);
                        if (b >= (unsigned long long)hi) {
                            more = false;
                            break;
                        }
                        pool = (int64_t)b;
                        pool_end = pool + C.fetch < hi ? pool + C.fetch : hi;
                        // streamed input: see trace_loop
                        if (C.ready && !wait_flag(C.ready + (pool_end - 1) / C.ready_chunk,
                                                  C.status, C.wait_polls)) {
                            if (lane == 0) atomicMax(counter, (unsigned long long)hi);
                            pool = pool_end;
                            more = false;
                            break;
                        }
                    }
                    const int64_t left = pool_end - pool;
                    const int take = left < 32 ? (int)left : 32;
                    bool ok = false;
                    WalkSeg w;
                    unsigned k = 0u;
                    if (lane < take) {
                        int64_t kk = pool + lane;
                        bool known = true;
                        if (C.order) {  // a caller's order: entries outside [0, nR) are skipped
                            kk = C.order[kk];
                            known = kk >= 0 && kk < C.nR;
                            if (!known) atomicCAS(C.status, 0, RSI_ERR_BAD_INDEX);
                        }
                        if (STATS) ++segs;
                        if (known) {
                            k = (unsigned)kk;
                            w.ax_ = C.A[3 * kk];
                            w.ay_ = C.A[3 * kk + 1];
                            w.az_ = C.A[3 * kk + 2];
                            const float bx = C.B[3 * kk], by = C.B[3 * kk + 1],
                                        bz = C.B[3 * kk + 2];
                            ok = finite3(w.ax_, w.ay_, w.az_) && finite3(bx, by, bz) &&
                                 start != kNoRoot;
                            w.dx = __fsub_rn(bx, w.ax_);
                            w.dy = __fsub_rn(by, w.ay_);
                            w.dz = __fsub_rn(bz, w.az_);
                            walk_axis(w.ax_, w.dx, w.ix, w.nx, w.fx);
                            walk_axis(w.ay_, w.dy, w.iy, w.ny, w.fy);
                            walk_axis(w.az_, w.dz, w.iz, w.nz, w.fz);
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
                const int n = min(avail, __popc(idle));
                const int r = __popc(idle & lt);
                if (cur == kDone && r < n) {
                    const float4 q0 = sg.q[0][head + r], q1 = sg.q[1][head + r];
                    const float4 q2 = sg.q[2][head + r], q3 = sg.q[3][head + r];
                    s.ax_ = q0.x;
                    s.ay_ = q0.y;
                    s.az_ = q0.z;
                    i = (unsigned)f2i(q0.w);
                    s.dx = q1.x;
                    s.dy = q1.y;
                    s.dz = q1.z;
                    s.fz = q1.w;
                    s.ix = q2.x;
                    s.iy = q2.y;
                    s.iz = q2.z;
                    s.nx = q2.w;
                    s.ny = q3.x;
                    s.nz = q3.y;
                    s.fx = q3.z;
                    s.fy = q3.w;
                    cur = start;
                    sp = 0;
                    count = 0;
                    best = kNoBest;
                    tlim = 1.f;
                }
                head += n;
                avail -= n;
                idle = __ballot_sync(FULL, cur == kDone);
                __syncwarp();  // every lane has read its entry before the next set-up
            }
            continue;
        }
        if (nl > 0 && (nd + nl >= kStall || dead + leaf == FULL ||
                       (!refillable && 4 * nl >= 32 - nd))) {
            // ---- triangle tests of the waiting leaves
            if (cur < 0 && cur != kDone) {
                s.range();
                const int pos0 = LEAFN ? (int)((unsigned)~cur >> 3) : ~cur;
                const int pos1 = LEAFN ? pos0 + (~cur & 7) : pos0;
                bool stop = false;
                for (int pos = pos0; pos <= pos1; ++pos) {
                    const float4* tp = C.tris + 3 * (int64_t)pos;
                    const float4 a = ld4(tp), b = ld4(tp + 1), c = ld4(tp + 2);
                    float t = 0.f, u = 0.f, v = 0.f, err = 0.f;
                    if (STATS) ++st.tests;
                    int r = mt32(s, a, b, c, MODE == RSI_MODE_NEAREST, t, u, v, err);
                    unsigned code = (unsigned)pos;
                    if (r == 2) {
                        if (STATS) ++st.fp64;
                        const float* pa = C.A + 3 * (int64_t)i;
                        const float* pb = C.B + 3 * (int64_t)i;
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
                        stop = true;
                        break;
                    }
                    if (MODE == RSI_MODE_COUNT) ++count;
                    if (MODE == RSI_MODE_NEAREST) {
                        bool take = best == kNoBest || t + err < tlo;
                        if (!take && !(t - err > tlim)) {
                            // the intervals overlap: compare the definition's
                            // t in FP64, ties to the lower triangle index
                            const int bpos = (int)(best & ~kBest64);
                            const double tn = exact_t(C.A, C.B, i, C.tris, pos);
                            const double tb = exact_t(C.A, C.B, i, C.tris, bpos);
                            take = tn < tb || (tn == tb && f2i(a.w) <
                                                   f2i(ld4(C.tris + 3 * (int64_t)bpos).w));
                        }
                        if (take) {
                            best = code;
                            tlo = t - err;
                            tlim = fminf(1.f, t + err);
                        }
                    }
                }
                if (MODE == RSI_MODE_BOOL && stop)
                    cur = kDone;
                else
                    cur = stack[sp--];
            }
            continue;
        }
        // ---- node steps until kStall lanes (a quarter of those left at the
        // end of the work) have none
        const int alive = refillable ? 32 : 32 - nd;
        const int floor_ = alive - (refillable ? kStall : max(1, (alive + 3) / 4));
        do {
            if (cur >= 0) {
                ulonglong2 q0, q1, q2;
                int4 rc;
                ld_node(C.nodes + 4 * (int64_t)cur, q0, q1, q2, rc);
                if (STATS) ++st.visits;
                const float2 lx = up2(q0.x), ly = up2(q0.y), lz = up2(q1.x);
                const float2 hx = up2(q1.y), hy = up2(q2.x), hz = up2(q2.y);
                float t0, t1;
                const bool h0 = walk_box<MODE == RSI_MODE_NEAREST>(s, lx.x, ly.x, lz.x, hx.x, hy.x,
                                                                   hz.x, tlim, t0);
                const bool h1 = walk_box<MODE == RSI_MODE_NEAREST>(s, lx.y, ly.y, lz.y, hx.y, hy.y,
                                                                   hz.y, tlim, t1);
                const int x0 = walk_item<LEAFN>(rc.x, rc.z), x1 = walk_item<LEAFN>(rc.y, rc.w);
                if (h0 && h1) {
                    const bool near0 = t0 <= t1;
                    cur = near0 ? x0 : x1;
                    if (sp >= kWalkStack) {  // deeper than any tree: corrupt
                        atomicCAS(C.status, 0, RSI_ERR_INTERNAL);
                        cur = kDone;
                    } else {
                        stack[++sp] = near0 ? x1 : x0;
                    }
                } else if (h0 || h1) {
                    cur = h0 ? x0 : x1;
                } else {
                    cur = stack[sp--];
                }
            }
            if (++steps > bound) {
                if (lane == 0) atomicCAS(C.status, 0, RSI_ERR_INTERNAL);
                cur = kDone;
            }
        } while (__popc(__ballot_sync(FULL, cur >= 0)) > floor_);
    }
}

}  // namespace rsi
