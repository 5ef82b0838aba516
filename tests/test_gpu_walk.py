"""The phased traversal loop (default options) against the general loop (a
32-entry stack takes it), which the oracle tests check: every mode, leaf
sizes that change the leaf items, mesh sizes around one leaf and around a
node, segment counts around a warp, a set-up batch and a fetched chunk, and
segments that the set-up treats apart (non-finite, zero components, zero
length, far starts)."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def special(seg, rng):
    A, B = seg.A.copy(), seg.B.copy()
    n = A.shape[0]
    for k, f in enumerate(range(0, n, 7)):
        j = k % 6
        if k % 13 == 12:  # far longer than any mesh, on every axis
            A[f], B[f] = (-2e7, -1e7, -3e7), (2e7, 1e7, 3e7)
        elif j == 0:
            A[f, rng.integers(3)] = (np.nan, np.inf, -np.inf)[k % 3]
        elif j == 1:
            B[f] = A[f]
        elif j == 2:
            B[f, rng.integers(3)] = A[f, 0]
            A[f] = B[f]
            A[f, 2] -= 1
        elif j == 3:
            A[f] *= 1e6
        elif j == 4:
            A[f], B[f] = (0, 0, -3e38), (0, 0, 3e38)
        else:
            B[f] = A[f] + np.float32(1e-20)
    return A, B


def compare(bvh, A, B, **kw):
    for mode in ("bool", "count", "nearest"):
        got = bvh.intersect(A, B, mode, **kw)
        ref = bvh.intersect(A, B, mode, launch={"stack_depth": 32}, **kw)
        torch.cuda.synchronize()
        n = int(ref["n_hits"].item()) if "n_hits" in ref else None
        for k in ref:
            if k in ("flag", "count", "tri", "n_hits"):
                assert torch.equal(got[k], ref[k]), (mode, k)
            elif k in ("tuv", "point", "dist"):
                assert torch.all((got[k] - ref[k]).abs() <= 2e-5 * ref[k].abs().clamp(min=1)), k
            elif k == "hit_idx":
                assert torch.equal(got[k][:n].sort()[0], ref[k][:n].sort()[0]), mode
    assert bvh.status() == 0


@pytest.mark.parametrize("n_tri", [1, 2, 3, 8, 9, 500])
@pytest.mark.parametrize("leaf", [1, 3, 8])
@pytest.mark.parametrize("n_seg", [1, 31, 33, 1000])
def test_small_meshes(n_tri, leaf, n_seg):
    rng = np.random.default_rng(n_tri * 1000 + leaf * 100 + n_seg)
    mesh, seg = synth.random_soup(rng, n_tri, n_seg)
    A, B = special(seg, rng)
    compare(rsi.BVH(dev(mesh.V), dev(mesh.T), leaf_size=leaf), dev(A), dev(B))


@pytest.mark.parametrize("n_seg", [4097, 70_001])
def test_terrain_compaction_and_order(n_seg):
    mesh, seg, _ = synth.workload_diff(seed=8, n_seg=n_seg, G=65)
    A, B = special(seg, np.random.default_rng(n_seg))
    bvh = rsi.BVH(dev(mesh.V), dev(mesh.T))
    A, B = dev(A), dev(B)
    compare(bvh, A, B, compact=True)
    order = bvh.segment_order(A, B)
    for mode, key in (("bool", "flag"), ("count", "count"), ("nearest", "tri")):
        a = bvh.intersect(A, B, mode)[key]
        b = bvh.intersect(A, B, mode, launch={"order": order})[key]
        assert torch.equal(a, b), mode
    assert bvh.status() == 0


@pytest.mark.parametrize("far", [10.0, 1e5])
def test_detail_in_a_far_larger_mesh(far):
    """A fine terrain beside one triangle `far` away: the nodes' grid blurs the
    terrain's boxes (10: still fine; 1e5: most leaves are below a grid step,
    and the loop reads the exact nodes)."""
    mesh, seg, _ = synth.workload_diff(seed=9, n_seg=5000, G=65)
    n = mesh.V.shape[0]
    V = np.concatenate([mesh.V, np.float32(far) + np.eye(3, dtype=np.float32)]).astype(np.float32)
    T = np.concatenate([mesh.T, [[n, n + 1, n + 2]]]).astype(np.int32)
    A, B = special(seg, np.random.default_rng(1))
    bvh = rsi.BVH(dev(V), dev(T))
    compare(bvh, dev(A), dev(B))
    ref = bvh.intersect(dev(A), dev(B), "nearest", stats=True)["stats"]
    # no more nodes than the general loop's binary ones, but for the pads
    gen = bvh.intersect(dev(A), dev(B), "nearest", stats=True, launch={"stack_depth": 32})["stats"]
    assert ref["node_visits"] <= 1.01 * gen["node_visits"]
    V[:n, 2] += np.float32(0.01)
    bvh.refit(dev(V))
    compare(bvh, dev(A), dev(B))
    compare(bvh, dev(A), dev(B), compact=True)


def test_packets_on_the_same_nodes():
    for far in (None, 1e5):
        mesh, seg, _ = synth.workload_diff(seed=10, n_seg=3001, G=33)
        V, T = mesh.V, mesh.T
        if far:
            V = np.concatenate([V, np.float32(far) + np.eye(3)]).astype(np.float32)
            T = np.concatenate([T, [[len(V) - 3, len(V) - 2, len(V) - 1]]]).astype(np.int32)
        A, B = (dev(x) for x in special(seg, np.random.default_rng(2)))
        for leaf in (1, 4):
            bvh = rsi.BVH(dev(V), dev(T), leaf_size=leaf)
            for mode, key in (("bool", "flag"), ("count", "count"), ("nearest", "tri")):
                a = bvh.intersect(A, B, mode, launch={"packet": 1})[key]
                b = bvh.intersect(A, B, mode, launch={"stack_depth": 32})[key]
                assert torch.equal(a, b), (far, leaf, mode)
            assert bvh.status() == 0
