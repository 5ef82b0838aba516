"""The build's large sorts (2^18 keys and more: tiles ordered in shared memory
before they are written) and its centroids kept between two kernels: sizes
around the switch and a partial last tile, duplicate Morton codes, triangles
that are skipped, against a stable sort of the definition's codes."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def codes_of(V, T):
    """Morton codes by the definition (float32, Sec. 2); 0 for skipped ones."""
    F = np.float32
    P = V[T]
    ok = np.isfinite(P).all(axis=(1, 2))
    with np.errstate(all="ignore"):
        c = (((P[:, 0] + P[:, 1]).astype(F) + P[:, 2]).astype(F) / F(3)).astype(F)
    lo, hi = c[ok].min(0), c[ok].max(0)
    with np.errstate(all="ignore"):
        q = np.floor(((c - lo) / (hi - lo)).astype(F) * F(1024))
        q = np.clip(np.where(ok[:, None], q, 0), 0, 1023).astype(np.uint32)
    code = np.zeros(len(T), np.uint32)
    for b in range(10):
        for k in range(3):
            code |= ((q[:, k] >> b) & 1) << np.uint32(3 * b + 2 - k)
    return np.where(ok, code, 0).astype(np.uint32)


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1, 300_001])
@pytest.mark.parametrize("spread", [1.0, 0.004])  # 0.004: many triangles share a code
def test_order_is_the_stable_sort(n, spread):
    rng = np.random.default_rng(n)
    nv = 20_000
    V = (rng.uniform(0, 1, (nv, 3)) * spread).astype(np.float32)
    V[:2] = [[0, 0, 0], [1, 1, 1]]
    T = rng.integers(0, nv, (n, 3)).astype(np.int32)
    V[7] = np.nan
    T[0], T[1] = (0, 0, 0), (1, 1, 1)
    want = codes_of(V, T)
    bvh = rsi.BVH(torch.from_numpy(V).to(DEV), torch.from_numpy(T).to(DEV))
    g = bvh.export()
    order = np.argsort(want, kind="stable")
    np.testing.assert_array_equal(g["order"], order)
    np.testing.assert_array_equal(g["codes"], want[order])
    assert bvh.status() == 0


@pytest.mark.parametrize("n", [2047, 262_144, 262_145, 600_001])
def test_large_segment_orders(n):
    rng = np.random.default_rng(n)
    V = torch.rand(300, 3, device=DEV)
    T = torch.from_numpy(rng.integers(0, 300, (500, 3)).astype(np.int32)).to(DEV)
    bvh = rsi.BVH(V, T)
    A = torch.from_numpy(rng.uniform(-1, 2, (n, 3)).astype(np.float32)).to(DEV)
    B = A.clone()  # midpoint and octant: repeated segments share a key
    m = n // 2
    A[m:2 * m] = A[:m].clone()
    B[m:2 * m] = B[:m].clone()
    o = bvh.segment_order(A, B).long().cpu().numpy()
    assert np.array_equal(np.sort(o), np.arange(n))
    pos = np.empty(n, np.int64)
    pos[o] = np.arange(n)
    # stable: of two segments with one key the earlier comes first
    assert np.all(pos[:m] < pos[m:2 * m])
