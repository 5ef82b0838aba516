"""A mesh with a small part of its triangles in a patch far below a step of the
four-way nodes' grid: the walk of a segment aimed at the patch may not grow
with the triangles per grid cell.  Compared with the general loop, which reads
the exact binary nodes (a 32-entry stack takes it).

Bounds, from the rule (kBlurRatio): leaf boxes that stay on the grid are met at
most 2.5 times as often as the exact ones over all directions, 4 times for
these; with twice the boxes per step, 1.5 times the node visits."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

from test_gpu_walk import compare, dev

pytestmark = pytest.mark.gpu


def patched(size, p, G=129):
    """A terrain (2 (G-1)^2 triangles) and below it a terrain of 2 (p-1)^2
    triangles, `size` wide; segments through the small one."""
    big = synth.workload_diff(seed=21, n_seg=8, G=G)[0]
    small = synth.workload_diff(seed=22, n_seg=8, G=p)[0]
    Vb = big.V.copy()
    Vb[:, 2] += 1
    V = np.concatenate([Vb, small.V * np.float32(size)]).astype(np.float32)
    T = np.concatenate([big.T, small.T + len(Vb)]).astype(np.int32)
    rng = np.random.default_rng(23)
    xy = rng.uniform(0.02, 0.98, (4000, 2))
    A = np.column_stack([xy, np.full(4000, -0.5)]) * size
    B = np.column_stack([xy + rng.normal(0, 0.02, (4000, 2)), np.full(4000, 0.5)]) * size
    return V, T, A.astype(np.float32), B.astype(np.float32)


@pytest.mark.parametrize("p", [9, 33, 45])  # 0.4, 6 and 11 % of the triangles
@pytest.mark.parametrize("size", [1e-5, 1e-4, 1e-3, 3e-3])
@pytest.mark.parametrize("leaf", [1, 4])
def test_detail_in_a_small_part(size, p, leaf):
    V, T, A, B = patched(size, p)
    bvh = rsi.BVH(dev(V), dev(T), leaf_size=leaf)
    A, B = dev(A), dev(B)
    compare(bvh, A, B)
    for mode in ("count", "nearest"):
        got = bvh.intersect(A, B, mode, stats=True)["stats"]
        gen = bvh.intersect(A, B, mode, stats=True, launch={"stack_depth": 32})["stats"]
        if p == 9:  # 128 leaves: at most three groups below the limit
            assert got["tri_tests"] <= 127 * 4000
            continue
        assert got["tri_tests"] <= 4 * gen["tri_tests"], (mode, got, gen)
        assert got["node_visits"] <= 1.5 * gen["node_visits"], (mode, got, gen)


def test_refit_moves_the_line():
    """The rule follows the boxes of a refit, both ways, on one handle."""
    V, T, A, B = patched(0.3, 33)
    n = len(V) - 33 * 33
    small = V.copy()
    small[n:] *= np.float32(1e-4)
    bvh = rsi.BVH(dev(V), dev(T))
    for v, scale in ((V, 1.0), (small, 1e-4), (V, 1.0)):
        bvh.refit(dev(v))
        a, b = dev(A * np.float32(scale)), dev(B * np.float32(scale))
        compare(bvh, a, b)
        got = bvh.intersect(a, b, "nearest", stats=True)["stats"]
        gen = bvh.intersect(a, b, "nearest", stats=True, launch={"stack_depth": 32})["stats"]
        assert got["tri_tests"] <= 4 * gen["tri_tests"]


def test_ordinary_meshes_stay_on_the_grid():
    """Fewer node visits than binary nodes take: the four-way records serve."""
    for mesh, seg in (synth.workload_diff(seed=9, n_seg=5000, G=129)[:2],
                      synth.random_soup(np.random.default_rng(3), 5000, 5000)):
        bvh = rsi.BVH(dev(mesh.V), dev(mesh.T))
        A, B = dev(seg.A), dev(seg.B)
        got = bvh.intersect(A, B, "count", stats=True)["stats"]
        gen = bvh.intersect(A, B, "count", stats=True, launch={"stack_depth": 32})["stats"]
        assert got["node_visits"] <= 0.75 * gen["node_visits"]
