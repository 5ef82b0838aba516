"""The work a user has this package do, as timed cases.

A case is a dict of plain values.  ``kind`` says which call it is:

* ``query``   segments against a tree that the program keeps (``BVH.intersect``)
* ``step``    the mesh moved too far for a refit: rebuild, then query
* ``train``   one fitting step on a kept tree: refit, differentiable nearest
              crossing, gradients of vertices and segment ends
* ``fit``     the same without a kept tree (``nearest_hit(V, T, A, B)``)
* ``ordered`` coherent segment order, then a nearest query in that order
* ``inside``  odd-parity inside test of points against a closed mesh
* ``host``    segments in pinned host memory, flags back on the host
* ``batch``   many meshes with their own segments, built and traversed at once

Meshes are the terrains and closed star-shaped surfaces of the package's own
workloads (``synth.py``): a ``G`` x ``G`` height field, or an icosphere of
``level`` subdivisions.  Segments are drawn as there: ``random`` (start in the
grown mesh box, any direction, length log-uniform in [0.01, 1]), ``vertical``
(near-vertical, through the terrain), ``raster`` (exactly vertical, a pixel
grid), ``band`` (from below to above the terrain's mean plane) and ``cube``
(both ends uniform in a cube around a closed surface).
"""
import functools
import math

import numpy as np
import torch

import paper_2209_02878_gb300 as rsi
from paper_2209_02878_gb300 import synth

_DEV = "cuda:0"


def listed():
    return [
        # a few thousand segments of an interactive tool against a small mesh:
        # launch latency and host work
        dict(name="small_bool", kind="query", mesh="terrain", G=32, segs="band", mode="bool",
             n=10000),
        # the paper's experiment: tree and crossing flags of 10M random segments
        dict(name="paper_step", kind="step", mesh="terrain", G=123, segs="random", mode="bool",
             n=10000000),
        # crossing counts against a large closed surface (tree larger than L2)
        dict(name="sphere_count", kind="query", mesh="sphere", level=8, segs="cube",
             mode="count", n=1000000),
        # nearest crossings against the same
        dict(name="sphere_nearest", kind="query", mesh="sphere", level=8, segs="cube",
             mode="nearest", n=1000000),
        # an orthographic view: coherent vertical segments, one per pixel
        dict(name="raster_nearest", kind="query", mesh="terrain", G=123, segs="raster",
             mode="nearest", n=3163 * 3163),
        # fitting a terrain to measured rays: the tree is kept and refit
        dict(name="train_step", kind="train", mesh="terrain", G=257, segs="vertical", n=262144),
        # the same as a plain function of a mesh, nothing kept between calls
        dict(name="fit_fresh", kind="fit", mesh="terrain", G=102, segs="vertical", n=65537),
        # a large deforming surface: the rebuild outweighs the query
        dict(name="rebuild_large", kind="step", mesh="sphere", level=8, segs="cube",
             mode="nearest", n=100003),
        # fixed rays, sorted once for the queries that follow
        dict(name="ordered_nearest", kind="ordered", mesh="terrain", G=257, segs="vertical",
             n=1000003),
        # sampling a solid: which points lie inside
        dict(name="inside_points", kind="inside", mesh="sphere", level=6, n=1000003),
        # segments that arrive in host memory (a file, another process)
        dict(name="host_bool", kind="host", mesh="terrain", G=123, segs="random", n=4000037),
        # many objects at once, flags and nearest crossings mixed
        dict(name="batch_mixed", kind="batch", items=16, n_lo=10000, n_hi=1000000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "step", "step", "train", "fit", "ordered",
                       "inside", "host", "batch"])
    if kind == "batch":
        return dict(kind=kind, items=rng.randint(2, 24), n_lo=1000, n_hi=_log_int(rng, 3e4, 6e5))
    if kind == "inside":
        return dict(kind=kind, mesh="sphere", level=rng.randint(3, 7), n=_log_int(rng, 1e3, 1e6))
    if kind in ("train", "fit"):
        return dict(kind=kind, mesh="terrain", G=rng.randint(24, 320), segs="vertical",
                    n=_log_int(rng, 2e3, 5e5))
    if kind == "ordered":
        return dict(kind=kind, mesh="terrain", G=rng.randint(48, 320), segs="vertical",
                    n=_log_int(rng, 2e4, 1.5e6))
    if kind == "host":
        return dict(kind=kind, mesh="terrain", G=rng.randint(32, 200), segs="random",
                    n=_log_int(rng, 2e4, 6e6))
    mode = rng.choice(["bool", "count", "nearest"])
    if rng.random() < 0.4:
        return dict(kind=kind, mesh="sphere", level=rng.randint(3, 8), segs="cube", mode=mode,
                    n=_log_int(rng, 1e4, 1e6))
    segs = rng.choice(["random", "vertical", "raster", "band"])
    top = {"random": 6e6, "vertical": 1e6, "raster": 6e6, "band": 2e6}[segs]
    n = _log_int(rng, 1e4, top)
    if segs == "raster":
        n = int(math.isqrt(n)) ** 2
    return dict(kind=kind, mesh="terrain", G=rng.randint(24, 320), segs=segs, mode=mode, n=n)


# ------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=16)
def _ico(level):
    U, T = synth.icosphere_topology(level)
    return U, T.astype(np.int32)


def _terrain(G, seed):
    m = synth.heightfield(G, np.random.default_rng(seed))
    return torch.from_numpy(m.V).to(_DEV), torch.from_numpy(m.T).to(_DEV)


def _sphere(level, seed):
    """Star-shaped closed surface: smooth waves of the radius and a little
    noise, below the edge length."""
    U, T = _ico(level)
    rng = np.random.default_rng(seed)
    w = rng.normal(0.0, 1.0, (3, 6)) * np.array([2.0, 3.0, 4.0, 5.0, 7.0, 9.0])
    r = 1.0 + 0.012 * np.sin(U @ w + rng.uniform(0, 2 * math.pi, 6)).sum(1)
    r += rng.normal(0.0, 0.1 / 2 ** level, U.shape[0])
    V = (U * r[:, None]).astype(np.float32)
    return torch.from_numpy(V).to(_DEV), torch.from_numpy(T).to(_DEV)


def _mesh(case, seed):
    if case["mesh"] == "terrain":
        return _terrain(case["G"], seed)
    return _sphere(case["level"], seed)


def _gen(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(seed)
    return g


def _uniform(g, n, lo, hi):
    lo = torch.as_tensor(lo, dtype=torch.float32, device=_DEV)
    hi = torch.as_tensor(hi, dtype=torch.float32, device=_DEV)
    return lo + (hi - lo) * torch.rand(n, 3, device=_DEV, generator=g)


def _segments(segs, n, V, seed):
    g = _gen(seed)
    if segs == "random":
        lo, hi = V.amin(0), V.amax(0)
        ext = hi - lo
        A = _uniform(g, n, lo - 0.1 * ext, hi + 0.1 * ext)
        d = torch.randn(n, 3, device=_DEV, generator=g)
        d /= d.norm(dim=1, keepdim=True)
        u = torch.rand(n, 1, device=_DEV, generator=g)
        return A, A + d * torch.exp(math.log(0.01) * (1.0 - u))
    if segs == "vertical":
        xy = 0.02 + 0.96 * torch.rand(n, 2, device=_DEV, generator=g)
        dxy = 0.02 * torch.randn(n, 2, device=_DEV, generator=g)
        one = torch.ones(n, 1, device=_DEV)
        return torch.cat([xy, -one], 1), torch.cat([xy + dxy, one], 1)
    if segs == "raster":
        k = math.isqrt(n)
        # the view is shifted by a fraction of a pixel from input to input
        off = np.random.default_rng(seed).uniform(0.25, 0.75, 2)
        i = torch.arange(n, device=_DEV)
        x = ((i % k).double() + off[0]) / k
        y = ((i // k).double() + off[1]) / k
        one = torch.ones(n, device=_DEV)
        return (torch.stack([x.float(), y.float(), -one], 1),
                torch.stack([x.float(), y.float(), one], 1))
    if segs == "band":
        return (_uniform(g, n, [0, 0, -0.5], [1, 1, 0]), _uniform(g, n, [0, 0, 0], [1, 1, 0.5]))
    c = [1.5, 1.5, 1.5]
    m = [-1.5, -1.5, -1.5]
    return _uniform(g, n, m, c), _uniform(g, n, m, c)


def _moved(V, mesh, seed):
    """The vertices after a training step: a small move along the height."""
    g = _gen(seed + 1)
    dz = 0.002 * torch.randn(V.shape[0], device=_DEV, generator=g)
    W = V.clone()
    W[:, 2] += dz
    return W


def _batch_items(case, seed):
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(case["items"])  # sizes are the case's, values the seed's
    items = []
    for k in range(case["items"]):
        nt = math.exp(sizes.uniform(math.log(1e3), math.log(2e5)))
        n = int(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        sub = int(rng.integers(1 << 30))
        if k % 2 == 0:
            V, T = _terrain(max(2, int(round(math.sqrt(nt / 2.0))) + 1), sub)
            A, B = _segments("random", n, V, sub)
            items.append((V, T, A, B, "bool"))
        else:
            lev = min((3, 4, 5, 6), key=lambda q: abs(math.log(20 * 4 ** q) - math.log(nt)))
            V, T = _sphere(lev, sub)
            A, B = _segments("cube", n, V, sub)
            items.append((V, T, A, B, "nearest"))
    return items


def _inputs(case, seed):
    V, T = _mesh(case, seed)
    if case["kind"] == "inside":
        return V, T, _uniform(_gen(seed), case["n"], [-1.2] * 3, [1.2] * 3), None
    A, B = _segments(case["segs"], case["n"], V, seed)
    return V, T, A, B


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(kind=kind, batch=rsi.Batch(_batch_items(case, seed)))
    V, T, A, B = _inputs(case, seed)
    s = dict(kind=kind, mode=case.get("mode"), V=V, T=T, A=A, B=B)
    if kind == "fit":
        s["leaves"] = [x.clone().requires_grad_(True) for x in (V, A, B)]
    elif kind == "train":
        s["bvh"] = rsi.BVH(V, T)
        W = _moved(V, case["mesh"], seed)
        s["leaves"] = [x.clone().requires_grad_(True) for x in (W, A, B)]
    else:
        s["bvh"] = rsi.BVH(V, T)
    if kind in ("train", "fit"):
        s["w"] = torch.randn(case["n"], 3, device=_DEV, generator=_gen(seed + 2))
    if kind == "host":
        s["A"], s["B"] = A.cpu().pin_memory(), B.cpu().pin_memory()
        s["out"] = {"flag": torch.empty(case["n"], dtype=torch.uint8, pin_memory=True)}
    return s


def run(state):
    kind = state["kind"]
    if kind == "batch":
        return state["batch"].run_graph()
    if kind in ("train", "fit"):
        V, A, B = state["leaves"]
        bvh = state.get("bvh")
        if bvh is not None:
            bvh.refit(V.detach())
        P, tuv, tri = rsi.nearest_hit(V, state["T"], A, B, bvh=bvh)
        gV, gA, gB = torch.autograd.grad(P, (V, A, B), grad_outputs=state["w"])
        return dict(point=P.detach(), tuv=tuv.detach(), tri=tri, grad_V=gV, grad_A=gA, grad_B=gB)
    bvh = state["bvh"]
    if kind == "step":
        bvh.build(state["V"], state["T"])
    if kind in ("step", "query"):
        return bvh.intersect(state["A"], state["B"], state["mode"])
    if kind == "ordered":
        order = bvh.segment_order(state["A"], state["B"])
        out = bvh.intersect(state["A"], state["B"], "nearest", launch={"order": order})
        return dict(out, order=order)
    if kind == "inside":
        return bvh.points_inside(state["A"])
    return bvh.intersect_host(state["A"], state["B"], "bool", out=state["out"])


# --------------------------------------------------------------------- work
def _mesh_size(case):
    if case["mesh"] == "terrain":
        return case["G"] ** 2, 2 * (case["G"] - 1) ** 2
    return 10 * 4 ** case["level"] + 2, 20 * 4 ** case["level"]


_OUT = {"bool": 1, "count": 4, "nearest": 32}


def work(case):
    """Bytes: vertices, triangles, segments read once, results written once.
    Flops: one crossing test (50) and the box tests of one root-to-leaf path
    (20 each) per segment, and one adjoint (150) where there are gradients."""
    if case["kind"] == "batch":
        b = f = 0.0
        sizes = np.random.default_rng(case["items"])
        for k in range(case["items"]):
            nt = math.exp(sizes.uniform(math.log(1e3), math.log(2e5)))
            n = int(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
            b += 18 * nt + n * (24 + _OUT["bool" if k % 2 == 0 else "nearest"])
            f += n * (50 + 20 * math.log2(nt))
        return {"bytes": b, "flops": f}
    nv, nt = _mesh_size(case)
    n, kind = case["n"], case["kind"]
    b = 12 * nv + 12 * nt
    f = n * (50 + 20 * math.log2(nt))
    if kind in ("query", "step"):
        b += n * (24 + _OUT[case["mode"]])
    elif kind == "ordered":
        b += n * (24 + 32 + 4)
    elif kind == "inside":
        b += n * 13
    elif kind == "host":
        b += n * 25
    else:  # point, tuv, tri; upstream gradient in, three gradients out
        b += 12 * nv + n * (24 + 28 + 12 + 24)
        f += n * 150
    return {"bytes": float(b), "flops": float(f)}


# -------------------------------------------------------------------- exact
def _cross(a, b):
    return torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1],
                        a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],
                        a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], 1)


def _dot(a, b):
    return a[:, 0] * b[:, 0] + a[:, 1] * b[:, 1] + a[:, 2] * b[:, 2]


def _terrain_nearest(V, T, A, B, G):
    """Nearest crossing of near-vertical segments with a G x G terrain, in 64
    bits: every segment is tested against the two triangles of each grid cell
    that the box of its (x, y) extent touches."""
    n = A.shape[0]
    best_t = torch.full((n,), math.inf, dtype=torch.float64, device=_DEV)
    best = torch.full((n,), -1, dtype=torch.int64, device=_DEV)
    uv = torch.zeros(n, 2, dtype=torch.float64, device=_DEV)
    eps = 1e-6
    lo = (torch.minimum(A, B)[:, :2].double() - eps) * (G - 1)
    hi = (torch.maximum(A, B)[:, :2].double() + eps) * (G - 1)
    c0 = lo.floor().long().clamp(0, G - 2)
    c1 = hi.floor().long().clamp(0, G - 2)
    span = c1 - c0
    sx, sy = int(span[:, 0].max()), int(span[:, 1].max())
    for dy in range(sy + 1):
        for dx in range(sx + 1):
            idx = ((span[:, 0] >= dx) & (span[:, 1] >= dy)).nonzero()[:, 0]
            if idx.numel() == 0:
                continue
            a, b = A[idx].double(), B[idx].double()
            d = b - a
            cell = (c0[idx, 1] + dy) * (G - 1) + c0[idx, 0] + dx
            for half in (0, 1):
                j = 2 * cell + half
                tv = T[j].long()
                v0, v1, v2 = (V[tv[:, k]].double() for k in range(3))
                e1, e2, s0 = v1 - v0, v2 - v0, a - v0
                p, q = _cross(d, e2), _cross(s0, e1)
                det = _dot(e1, p)
                sg = torch.where(det < 0, -1.0, 1.0).double()
                det, nu, nv, nt = sg * det, sg * _dot(s0, p), sg * _dot(d, q), sg * _dot(e2, q)
                hit = (det > 0) & (nu >= 0) & (nv >= 0) & (nu + nv <= det) & (nt >= 0) & (nt <= det)
                t = torch.where(hit, nt / det, math.inf)
                bt, bj = best_t[idx], best[idx]
                take = hit & ((t < bt) | ((t == bt) & (j < bj)))
                w = idx[take]
                best_t[w], best[w] = t[take], j[take]
                uv[w, 0], uv[w, 1] = (nu / det)[take], (nv / det)[take]
    hit = best >= 0
    t = torch.where(hit, best_t, torch.zeros_like(best_t))
    d = B.double() - A.double()
    point = torch.where(hit[:, None], A.double() + t[:, None] * d, torch.zeros_like(d))
    dist = t * d.norm(dim=1)
    return best, torch.cat([t[:, None], uv], 1), point, dist


def _terrain_grads(V, T, A, B, tri, w):
    """Gradients of sum(w . point) with the crossed triangle held fixed, in
    64 bits: with M = [-d, e1, e2] and M x = a - v0, x = (t, u, v)."""
    h = (tri >= 0).nonzero()[:, 0]
    tv = T[tri[h]].long()
    a, d = A[h].double(), B[h].double() - A[h].double()
    v0, v1, v2 = (V[tv[:, k]].double() for k in range(3))
    e1, e2, gp = v1 - v0, v2 - v0, w[h].double()
    c12, c20, c01 = _cross(e1, e2), _cross(e2, -d), _cross(-d, e1)
    det = _dot(-d, c12)
    x = [_dot(c, a - v0) / det for c in (c12, c20, c01)]
    lam = c12 * (_dot(gp, d) / det)[:, None]
    gA, gB = torch.zeros_like(A, dtype=torch.float64), torch.zeros_like(B, dtype=torch.float64)
    gV = torch.zeros_like(V, dtype=torch.float64)
    gA[h] = (1 - x[0])[:, None] * (gp + lam)
    gB[h] = x[0][:, None] * (gp + lam)
    gV.index_add_(0, tv[:, 0], -(1 - x[1] - x[2])[:, None] * lam)
    gV.index_add_(0, tv[:, 1], -x[1][:, None] * lam)
    gV.index_add_(0, tv[:, 2], -x[2][:, None] * lam)
    return gV, gA, gB


def exact(case, seed):
    """Nearest crossings and gradients over terrains under near-vertical
    segments, whose candidate triangles are known from the grid; elsewhere the
    outputs are whole numbers, or every segment against every triangle would
    take too long."""
    kind = case["kind"]
    if kind == "batch" or case.get("segs") not in ("vertical", "raster"):
        return None
    if kind in ("query", "step") and case["mode"] != "nearest":
        return None
    V, T, A, B = _inputs(case, seed)
    if kind == "train":
        V = _moved(V, case["mesh"], seed)
    tri, tuv, point, dist = _terrain_nearest(V, T, A, B, case["G"])
    if kind in ("train", "fit"):
        w = torch.randn(case["n"], 3, device=_DEV, generator=_gen(seed + 2))
        gV, gA, gB = _terrain_grads(V, T, A, B, tri, w)
        return dict(point=point, tuv=tuv, tri=None, grad_V=gV, grad_A=gA, grad_B=gB)
    out = dict(tri=None, tuv=tuv, point=point, dist=dist)
    return dict(out, order=None) if kind == "ordered" else out
