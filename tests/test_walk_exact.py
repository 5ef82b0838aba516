"""The phased traversal's box test on the exact nodes carries no pad in the
mesh's own units (csrc/walk.cuh, walk_axis): on the CPU it still never rejects a
touched box, on the GPU a mesh that reads the exact nodes takes the same walk
at every scale."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

from test_slab_bound import touching_cases
from test_walk_box import edge_cases, walk32


@pytest.mark.parametrize("seed", range(3))
def test_touched_exact_boxes_are_never_rejected(seed):
    rng = np.random.default_rng(700 + seed)
    for A, B, LO, HI in (touching_cases(rng, 20_000), edge_cases(rng)):
        for ulp in (-1, 0, 1):
            miss = np.nonzero(~walk32(A, B, LO, HI, np.full(A.shape, ulp), unit=0.0))[0]
            assert miss.size == 0, (ulp, A[miss[:3]], B[miss[:3]])


@pytest.mark.gpu
@pytest.mark.parametrize("packet", [0, 1])
def test_the_walk_does_not_depend_on_the_scale(packet):
    """A terrain beside one triangle 1e5 of its sizes away, scaled as a whole by
    powers of two: the nodes' boxes, segments and hits scale exactly, and so
    must the counts of visits and tests (bound: 1.2 of the largest scale's, for
    the decisions that the pads turn)."""
    dev = torch.device("cuda:0")
    mesh, seg, _ = synth.workload_diff(seed=31, n_seg=4000, G=65)
    n = len(mesh.V)
    V = np.concatenate([mesh.V, 1e5 + np.eye(3)]).astype(np.float32)
    T = np.concatenate([mesh.T, [[n, n + 1, n + 2]]]).astype(np.int32)
    ref = None
    for k in (0, -17, -24):
        s = np.float32(2.0 ** k)
        bvh = rsi.BVH(torch.from_numpy(V * s).to(dev), torch.from_numpy(T).to(dev))
        A, B = (torch.from_numpy(x * s).to(dev) for x in (seg.A, seg.B))
        o = bvh.intersect(A, B, "count", stats=True, launch={"packet": packet})
        assert bvh.status() == 0
        if ref is None:
            ref = o
            continue
        assert torch.equal(o["count"], ref["count"])
        for key in ("node_visits", "tri_tests"):
            assert o["stats"][key] <= 1.2 * ref["stats"][key], (k, key)
