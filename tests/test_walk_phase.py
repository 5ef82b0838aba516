"""CPU check that the phased traversal's step bound ends a walk over a corrupt
tree whatever its phases do: csrc/walk_phase.h (the rules that the kernels
compile) drives an emulated warp over a cyclic tree.  With a leaf beside the
cycle each node phase ends after one step, with none it never leaves the node
phase."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2209_02878_gb300", "csrc")

# Lane k enters the root, a record of {itself} and, when k < leaves, a leaf that
# is tested first; lanes from `lanes` on have no segment.  Prints the node
# steps taken until the bound ends the walk (0: beyond `cap`).
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "walk_phase.h"
#ifdef UNCOUNTED  // a planted mistake: a phase of one step is not counted
static bool more(unsigned& left, int inner, int floor_) {
    return inner > floor_ && --left != 0u;
}
#else
static bool more(unsigned& left, int inner, int floor_) {
    return rsi::walk_more(left, inner, floor_);
}
#endif
int main(int, char** v) {
    const int lanes = atoi(v[1]), leaves = atoi(v[2]), stall = atoi(v[3]), visits = atoi(v[4]);
    enum { NODE, LEAF, DONE } cur[32];
    for (int k = 0; k < 32; ++k) cur[k] = k < lanes ? NODE : DONE;
    const unsigned bound = rsi::walk_bound(visits);
    const unsigned long long cap = 4ull * bound;
    unsigned left = bound;
    unsigned long long taken = 0;
    while (true) {
        int nd = 0, nl = 0;
        for (int k = 0; k < 32; ++k) { nd += cur[k] == DONE; nl += cur[k] == LEAF; }
        switch (rsi::walk_phase(nd, nl, false, stall)) {
        case rsi::kPhaseRefill:  // every lane is finished
            printf("%llu %u\n", taken, bound);
            return 0;
        case rsi::kPhaseLeaves:
            for (int k = 0; k < 32; ++k) if (cur[k] == LEAF) cur[k] = NODE;  // popped
            break;
        case rsi::kPhaseSteps: {
            const int floor_ = rsi::walk_floor(nd, false, stall);
            int inner;
            do {
                if (++taken > cap) { printf("0 %u\n", bound); return 0; }
                inner = 0;
                for (int k = 0; k < 32; ++k) {
                    if (cur[k] == NODE && k < leaves) cur[k] = LEAF;
                    inner += cur[k] == NODE;
                }
            } while (more(left, inner, floor_));
            if (left == 0u) for (int k = 0; k < 32; ++k) cur[k] = DONE;
        }
        }
    }
}
"""


def harness(tmp, *flags):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp / "walk.cpp", tmp / ("walk" + "".join(flags))
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + CSRC, *flags, str(src), "-o", str(exe)],
                   check=True)

    def run(*args):
        out = subprocess.run([str(exe), *map(str, args)], check=True, capture_output=True,
                             text=True, timeout=60).stdout
        return tuple(int(x) for x in out.split())
    return run


CASES = [(lanes, leaves, stall, visits)
         for lanes in (1, 2, 17, 32) for leaves in (0, 1, lanes // 2, lanes)
         for stall in (16, 20) for visits in (3, 1000)]


def test_a_cycle_ends_within_the_bound(tmp_path):
    run = harness(tmp_path)
    for case in CASES:
        taken, bound = run(*case)
        assert 0 < taken <= bound, case


def test_an_uncounted_step_never_ends(tmp_path):
    run = harness(tmp_path, "-DUNCOUNTED")
    assert run(32, 32, 16, 1000)[0] == 0


def test_every_lane_has_a_phase(tmp_path):
    """A correct walk takes a step, tests a leaf or refills: no phase without
    a lane to run it, and a step phase always takes a step."""
    src = tmp_path / "phase.cpp"
    src.write_text(r"""
#include "walk_phase.h"
int main() {
    for (int stall = 16; stall <= 20; stall += 4)
        for (int r = 0; r < 2; ++r)
            for (int nd = 0; nd <= 32; ++nd)
                for (int nl = 0; nl + nd <= 32; ++nl) {
                    const int inner = 32 - nd - nl;
                    const auto p = rsi::walk_phase(nd, nl, r, stall);
                    if (p == rsi::kPhaseRefill && nd == 0) return 1;
                    if (p == rsi::kPhaseLeaves && nl == 0) return 2;
                    if (p == rsi::kPhaseSteps && inner == 0) return 3;
                    if (p == rsi::kPhaseSteps && rsi::walk_floor(nd, r, stall) >= 32 - nd) return 4;
                }
    return 0;
}
""")
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    exe = tmp_path / "phase"
    subprocess.run([cxx, "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
