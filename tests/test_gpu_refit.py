"""Refits in a row without a synchronisation: the box pass starts while the
bounds pass still runs and waits for the grid of the moved vertices, so each
traversal between two refits must see that refit's grid and boxes and no other.
Vertex sets of very different sizes alternate (a stale grid would lose or
multiply hits), on one stream with a second handle in between, and as a graph."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def case(n_tri, seed, scales):
    """A soup of n_tri triangles at each scale with segments of that scale, and
    what the general loop finds on a tree built for it."""
    mesh, seg = synth.random_soup(np.random.default_rng(seed), n_tri, 3000)
    T, out = dev(mesh.T), []
    for k, s in enumerate(scales):
        shift = np.float32(s * k)
        V, A, B = (dev(x * np.float32(s) + shift) for x in (mesh.V, seg.A, seg.B))
        want = rsi.BVH(V, T).intersect(A, B, "nearest", launch={"stack_depth": 32})["tri"]
        out.append((V, A, B, want))
    return T, out


@pytest.mark.parametrize("n_tri", [1, 2, 511, 512, 513, 5000, 60_000])
@pytest.mark.parametrize("leaf", [1, 4])
def test_refits_in_a_row(n_tri, leaf):
    T, sets = case(n_tri, n_tri, (1.0, 1e3, 2e-3))
    U, other = case(700, 1, (0.5, 40.0, 3e-2))
    a = rsi.BVH(sets[0][0], T, leaf_size=leaf)
    b = rsi.BVH(other[0][0], U)
    got = []
    for r in range(12):
        (V, A, B, _), (W, C, D, _) = sets[r % 3], other[(r + 1) % 3]
        a.refit(V)
        b.refit(W)
        got.append((a.intersect(A, B, "nearest")["tri"], b.intersect(C, D, "nearest")["tri"]))
    for r, (x, y) in enumerate(got):
        assert torch.equal(x, sets[r % 3][3]), r
        assert torch.equal(y, other[(r + 1) % 3][3]), r
    assert a.status() == 0 and b.status() == 0


@pytest.mark.parametrize("n_tri", [513, 60_000])
def test_refits_in_a_graph(n_tri):
    T, sets = case(n_tri, n_tri, (1.0, 1e3, 2e-3))
    bvh = rsi.BVH(sets[0][0], T)
    outs = [bvh.intersect(A, B, "nearest") for _, A, B, _ in sets]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for (V, A, B, _), o in zip(sets, outs):
            bvh.refit(V)
            bvh.intersect(A, B, "nearest", out=o)
    for _ in range(5):
        for o in outs:
            o["tri"].fill_(-7)
        g.replay()
        for o, (_, _, _, want) in zip(outs, sets):
            assert torch.equal(o["tri"], want)
    assert bvh.status() == 0
