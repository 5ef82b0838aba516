"""Block sizes in turn on one handle and one batch: from 512 threads on (736
for nearest) a block of the phased traversal takes more dynamic shared memory
than the default limit of 48 KB, so a smaller block between two larger ones
must leave the kernel's limit where the larger one needs it."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
KEY = {"bool": "flag", "count": "count", "nearest": "tri"}
BLOCKS = (1024, 640, 1024, 768, 32, 896, 1024)


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


# 2,000 segments are dealt out, 300,000 taken from the work counter
@pytest.mark.parametrize("n_seg", [2000, 300_000])
@pytest.mark.parametrize("leaf", [1, 3])
@pytest.mark.parametrize("mode", list(KEY))
def test_blocks_in_turn(mode, leaf, n_seg):
    mesh, seg = synth.random_soup(np.random.default_rng(5), 300, n_seg)
    A, B = dev(seg.A), dev(seg.B)
    bvh = rsi.BVH(dev(mesh.V), dev(mesh.T), leaf_size=leaf)
    want = bvh.intersect(A, B, mode)[KEY[mode]]
    for block in BLOCKS:
        got = bvh.intersect(A, B, mode, launch={"block_size": block})[KEY[mode]]
        assert torch.equal(got, want), block
    assert bvh.status() == 0


def test_batch_blocks_in_turn():
    rng = np.random.default_rng(6)
    items = []
    for mode in KEY:
        mesh, seg = synth.random_soup(rng, 200, 3000)
        items.append((dev(mesh.V), dev(mesh.T), dev(seg.A), dev(seg.B), mode))
    want = [rsi.BVH(V, T).intersect(A, B, m)[KEY[m]] for V, T, A, B, m in items]
    for block in BLOCKS:
        b = rsi.Batch(items, launch={"block_size": block})
        out = b.build().intersect()
        for o, w, it in zip(out, want, items):
            assert torch.equal(o[KEY[it[4]]], w), (block, it[4])
        assert b.status() == 0
        b.close()
