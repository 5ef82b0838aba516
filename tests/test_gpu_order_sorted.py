"""rsi_segment_order against a stable sort of its key (csrc/order.cu: Morton code
of the midpoint over the mesh's box grown by its extent, direction octant
below), recomputed in float32 on the host: the order must be that sort's, not
only a permutation.  Sizes on both sides of a tile, of the scan folded into the
scatter (31 tiles of 1,024), of the tiles ordered in shared memory (2^18) and
with a partial last tile; key widths of two, three and four digits; repeated
keys, midpoints outside the box and non-finite segments."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
F = np.float32


def sort_key(V, A, B, bits):
    """What the sort compares: the low 8 bits times the digits of the key."""
    p = (bits - 3) // 3
    levels = F(1 << p)
    lo, hi = V.min(0), V.max(0)
    code = np.zeros(len(A), np.uint64)
    octant = np.zeros(len(A), np.uint64)
    ok = np.ones(len(A), bool)
    with np.errstate(all="ignore"):
        for k in range(3):
            ext = np.maximum(F(hi[k] - lo[k]), F(1e-30))
            m = F(0.5) * (A[:, k] + B[:, k])
            x = (m - F(lo[k] - ext)) / F(F(3) * ext) * levels
            ok &= np.isfinite(x)
            q = np.where(ok, np.clip(x, F(0), levels - F(1)), 0).astype(np.uint64)
            for b in range(p):
                code |= ((q >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - k)
            octant |= (B[:, k] < A[:, k]).astype(np.uint64) << np.uint64(2 - k)
    key = np.where(ok, code << np.uint64(3) | octant, np.uint64(0xffffffff))
    digits = -(-(3 * p + 3) // 8)
    return key & np.uint64((1 << (8 * digits)) - 1)


@pytest.mark.parametrize("n", [1, 255, 1023, 1024, 1025, 31_744, 31_745, 32_768, 65_537, (1 << 18) - 1,
                               1 << 18, (1 << 18) + 1, 600_001])
@pytest.mark.parametrize("bits", [12, 24, 30])
def test_the_order_is_the_stable_sort_of_the_key(n, bits):
    rng = np.random.default_rng(n + bits)
    V = rng.uniform(0, 1, (300, 3)).astype(F)
    T = np.concatenate([np.arange(300).reshape(100, 3), rng.integers(0, 300, (400, 3))])
    A = rng.uniform(-2, 3, (n, 3)).astype(F)
    B = (A + rng.normal(0, 0.3, (n, 3))).astype(F)
    A[n // 3: n // 2] = A[0]
    B[n // 3: n // 2] = B[0]
    bad = rng.integers(0, n, max(1, n // 50))
    A[bad, rng.integers(0, 3, len(bad))] = rng.choice([np.nan, np.inf, -np.inf], len(bad))
    bvh = rsi.BVH(torch.from_numpy(V).to(DEV), torch.from_numpy(T.astype(np.int32)).to(DEV))
    got = bvh.segment_order(torch.from_numpy(A).to(DEV), torch.from_numpy(B).to(DEV), bits=bits)
    want = np.argsort(sort_key(V, A, B, bits), kind="stable")
    np.testing.assert_array_equal(got.cpu().numpy(), want)
