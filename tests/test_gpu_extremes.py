"""Every traversal against the oracle on meshes at the ends of the float range:
extents that overflow, near FLT_MAX, denormal, flat on one or two axes, a
single point, far from the origin, detail beside huge triangles, non-finite
vertices; built and refitted, with segments whose differences overflow."""
import numpy as np
import pytest
import torch

import oracle
import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth


pytestmark = pytest.mark.gpu
F = np.float32


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(torch.device("cuda:0"))


def soup(n_tri=400, n_seg=2000, seed=3):
    mesh, seg = synth.random_soup(np.random.default_rng(seed), n_tri, n_seg)
    return (x.astype(np.float64) - 0.5 for x in (mesh.V, seg.A, seg.B)), mesh.T


def scaled(s):
    (V, A, B), T = soup()
    return V * s, T, A * s, B * s


def flat(*axes):
    (V, A, B), T = soup()
    for k in axes:
        V[:, k] = 0.25
    return V, T, A, B


def shifted(o):
    (V, A, B), T = soup()
    return V + o, T, A + o, B + o


def beside(s):
    """A small soup, and triangles s times larger around and beside it."""
    (V, A, B), T = soup()
    W = np.random.default_rng(4).uniform(-s, s, (30, 3))
    return np.concatenate([V, W]), np.concatenate([T, np.arange(len(V), len(V) + 30).reshape(-1, 3)]), A, B


def holes():
    V, T, A, B = scaled(1.0)
    V[::7] = np.nan
    V[3::11, 1] = np.inf
    V[5::13] = -np.inf
    return V, T, A, B


CASES = {
    "denormal": lambda: scaled(2.0 ** -140), "2^-120": lambda: scaled(2.0 ** -120),
    "2^-70": lambda: scaled(2.0 ** -70), "2^70": lambda: scaled(2.0 ** 70),
    "2^100": lambda: scaled(2.0 ** 100), "2^126": lambda: scaled(2.0 ** 126),
    "extent overflows": lambda: scaled(6.7e38),
    "flat x": lambda: flat(0), "flat z": lambda: flat(2), "flat xy": lambda: flat(0, 1),
    "point": lambda: flat(0, 1, 2), "far": lambda: shifted(np.array([1e4, -3e3, 2e6])),
    "beside 1e3": lambda: beside(1e3), "beside 1e6": lambda: beside(1e6),
    "beside 3e38": lambda: beside(3e38), "holes": holes,
}


def inputs(name):
    with np.errstate(all="ignore"):
        V, T, A, B = (x.astype(np.int32) if k == 1 else x.astype(F)
                      for k, x in enumerate(CASES[name]()))
        # some segments from far away, along an axis, and of zero length
        A[:40] = A[:40] * F(64)
        B[40:80, 1:] = A[40:80, 1:]
        B[80:90] = A[80:90]
    return V, T, A, B


LAUNCHES = [{}, {"packet": 1}, {"stack_depth": 32}, {"stack_depth": 8}, {"node_width": 4},
            {"smem_nodes": 31}, {"sort_bits": 24}]


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("leaf", [1, 4])
@pytest.mark.parametrize("top", [0, 5])
def test_against_the_oracle(name, leaf, top):
    V, T, A, B = inputs(name)
    with np.errstate(all="ignore"):
        ref = oracle.brute(V, T, A, B)
    bvh = rsi.BVH(dev(V), dev(T), leaf_size=leaf, top_levels=top)
    A, B = dev(A), dev(B)
    for launch in LAUNCHES:
        for mode, key in (("bool", "flag"), ("count", "count"), ("nearest", "tri")):
            got = bvh.intersect(A, B, mode, launch=launch)[key].cpu().numpy()
            np.testing.assert_array_equal(got, ref[key], err_msg=f"{launch} {mode}")
    assert bvh.status() == 0


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("leaf", [1, 4])
def test_after_a_refit(name, leaf):
    V, T, A, B = inputs(name)
    half = V * F(0.5)
    A_, B_ = dev(A), dev(B)
    bvh = rsi.BVH(dev(V), dev(T), leaf_size=leaf)
    for W in (half, V):
        bvh.refit(dev(W))
        with np.errstate(all="ignore"):
            ref = oracle.brute(W, T, A, B)
        for mode, key in (("bool", "flag"), ("count", "count"), ("nearest", "tri")):
            got = bvh.intersect(A_, B_, mode)[key].cpu().numpy()
            np.testing.assert_array_equal(got, ref[key], err_msg=mode)
    assert bvh.status() == 0


@pytest.mark.parametrize("stack", [32, 64])
def test_a_batch_of_them(stack):
    its, want = [], []
    for k, name in enumerate(CASES):
        V, T, A, B = inputs(name)
        mode, key = (("bool", "flag"), ("count", "count"), ("nearest", "tri"))[k % 3]
        with np.errstate(all="ignore"):
            want.append((key, oracle.brute(V, T, A, B)[key]))
        its.append((dev(V), dev(T), dev(A), dev(B), mode))
    b = rsi.Batch(its, launch={"stack_depth": stack})
    for o, (key, w), name in zip(b.build().intersect(), want, CASES):
        np.testing.assert_array_equal(o[key].cpu().numpy(), w, err_msg=name)
    assert b.status() == 0
    b.close()
