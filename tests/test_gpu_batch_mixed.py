"""Batches that hold all three modes (a stream per mode) over meshes of every
kind that the phased loop treats apart: empty, one triangle, one leaf, coarse
for the nodes' grid (most leaves, and a small part of them), single segments,
at offsets that are no multiple of anything, with larger leaves and
with the general loop's stack; eager and as a graph, against single-mesh calls
on the general loop."""
import numpy as np
import pytest
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
KEY = {"bool": "flag", "count": "count", "nearest": "tri"}


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def terrain(seed, G, n_seg, far=None, patch=None):
    """A terrain, beside one triangle `far` away, or with a terrain `patch`
    wide below it (and the segments through that)."""
    mesh, seg, _ = synth.workload_diff(seed=seed, n_seg=n_seg, G=G)
    V, T, A, B = mesh.V, mesh.T, seg.A, seg.B
    if far:
        T = np.concatenate([T, [[len(V), len(V) + 1, len(V) + 2]]])
        V = np.concatenate([V, far + np.eye(3)])
    if patch:
        small, s2, _ = synth.workload_diff(seed=seed + 1, n_seg=n_seg, G=17)
        T = np.concatenate([T, small.T + len(V)])
        V = np.concatenate([V + np.array([0, 0, 1]), small.V * patch])
        A, B = s2.A * patch, s2.B * patch
    return V, T, A, B


def items():
    rng = np.random.default_rng(77)
    kinds = []
    for n_tri, n_seg in ((0, 300), (1, 1000), (7, 257), (8, 31), (9, 1), (500, 1), (1201, 3001)):
        mesh, seg = synth.random_soup(rng, n_tri, n_seg)
        kinds.append((mesh.V if n_tri else np.zeros((3, 3)), mesh.T, seg.A, seg.B))
    kinds += [terrain(41, 33, 2049), terrain(42, 33, 1500, far=1e5),
              terrain(43, 65, 1500, patch=1e-5)]
    out = []
    for k, (V, T, A, B) in enumerate(kinds):
        for q, mode in enumerate(KEY):
            cut = max(1, len(A) - 5 * ((k + q) % 3))
            out.append((dev(V.astype(np.float32)), dev(T.astype(np.int32).reshape(-1, 3)),
                        dev(A[:cut].astype(np.float32)), dev(B[:cut].astype(np.float32)), mode))
    return [out[i] for i in rng.permutation(len(out))]


@pytest.mark.parametrize("leaf", [1, 3, 8])
@pytest.mark.parametrize("stack", [32, 64])
@pytest.mark.parametrize("compact", [False, True])
def test_every_mode_and_mesh_in_one_batch(leaf, stack, compact):
    its = items()
    want = []
    for V, T, A, B, mode in its:
        bvh = rsi.BVH(V, T, leaf_size=leaf)
        want.append(bvh.intersect(A, B, mode, launch={"stack_depth": 32}))
    b = rsi.Batch(its, leaf_size=leaf, launch={"stack_depth": stack}, compact=compact)

    def check(what):
        torch.cuda.synchronize()
        for k, (o, w, it) in enumerate(zip(b.outputs, want, its)):
            key = KEY[it[4]]
            assert torch.equal(o[key], w[key]), (what, k, it[4])
            if it[4] == "nearest":
                for q in ("tuv", "point", "dist"):
                    lim = 2e-5 * w[q].abs().clamp(min=1)
                    assert torch.all((o[q] - w[q]).abs() <= lim), (what, k, q)
            if compact and it[4] != "bool":
                hits = torch.nonzero(w[key] >= 0 if it[4] == "nearest" else w[key] > 0).flatten()
                n = int(o["n_hits"].item())
                assert n == len(hits), (what, k)
                assert torch.equal(o["hit_idx"][:n].sort()[0].long(), hits), (what, k)
            o[key].fill_(77)
        assert b.status() == 0

    b.build().intersect()
    check("eager")
    b.intersect()
    check("eager again")
    for rebuild in (True, True, False):
        b.run_graph(rebuild=rebuild)
        check("graph")
    b.close()
