// Which phase a warp of the phased traversal (walk.cuh) runs next, and the
// bound that ends a walk over a corrupt tree.  Plain C++, so that the CPU tests
// drive the same rules.
#pragma once

#ifdef __CUDACC__
#define RSI_HD __host__ __device__ __forceinline__
#else
#define RSI_HD inline
#endif

namespace rsi {

// Once no segments are left to refill from, a phase runs for 1 / kTail of the
// lanes still at work.
constexpr int kTail = 4;

enum WalkPhase { kPhaseRefill, kPhaseLeaves, kPhaseSteps };

// nd finished lanes, nl lanes whose item is a leaf, the others (32 - nd - nl)
// with a node step; refillable: segments are left.
RSI_HD WalkPhase walk_phase(int nd, int nl, bool refillable, int stall) {
    if (nd == 32 || (refillable && nd >= nl && nd + nl >= stall)) return kPhaseRefill;
    if (nl > 0 && (nd + nl >= stall || nd + nl == 32 || (!refillable && kTail * nl >= 32 - nd)))
        return kPhaseLeaves;
    return kPhaseSteps;
}

// Node steps go on while more lanes than this have one.
RSI_HD int walk_floor(int nd, bool refillable, int stall) {
    if (refillable) return 32 - stall;
    const int tail = (31 + kTail - nd) / kTail;
    return (32 - nd) - (tail > 1 ? tail : 1);
}

// Node steps that a warp may take between two refills: each of its 32 segments
// takes at most max_visits, so more can only be a corrupt tree.
RSI_HD unsigned walk_bound(int max_visits) {
    return (unsigned)max_visits < 1u << 26 ? 32u * (unsigned)max_visits + 64u : 0xffffffffu;
}

// Counts the node step that left `inner` lanes with another one (left: steps
// that the bound still allows); whether the phase goes on.  Every step counts:
// a cycle through a leaf ends each phase after one step.
RSI_HD bool walk_more(unsigned& left, int inner, int floor_) {
    return --left != 0u && inner > floor_;
}

}  // namespace rsi
