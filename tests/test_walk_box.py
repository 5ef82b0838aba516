"""CPU check that the box test of the phased traversal (csrc/walk.cuh) never
rejects a box that the exact segment touches, over the same cases as the
general loop's test (tests/test_slab_bound.py): float32 emulations of the
per-axis constants (walk_axis) and of the clamped entry / exit parameters,
with the approximate reciprocal moved by -1, 0 and +1 ulp, on the exact
nodes' boxes and on the 15-bit grid of the four-way nodes (write_frame,
grid_axis).  CPU only."""
import numpy as np
import pytest

from test_slab_bound import slab32, touching_cases

F = np.float32


def fma32(a, b, c):
    # exact product in float64, one rounding there and one to float32
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def frame32(lo, hi):
    """Grid of a mesh box: per row origin and scale (write_frame)."""
    with np.errstate(all="ignore"):
        e = hi - lo
        widest = np.fmax(e.max(axis=1, keepdims=True), F(2.0 ** -80))
        return lo, (F(32760 / 32768) / np.fmax(e, widest * F(2.0 ** -20))).astype(F)


def grid32(lo, hi, o, s):
    """Faces of a box on the grid, as the decoded floats in [1, 2)."""
    with np.errstate(all="ignore"):
        a, b = (lo - o) * s * F(32768), (hi - o) * s * F(32768)
        q0 = np.fmin(np.fmax(np.floor(a - F(0.0625)), F(0)), F(32767))
        q1 = np.fmax(np.fmin(np.ceil(b + F(0.0625)), F(32767)), F(0))
        empty = lo > hi
        q0, q1 = np.where(empty, F(32767), q0), np.where(empty, F(0), q1)
    return (F(1) + q0 / F(32768)).astype(F), (F(1) + q1 / F(32768)).astype(F)


def walk32(a, b, lo, hi, rcp_ulp, grid=None, rel=2.0 ** -21, unit=2.0 ** -22, add=2.0 ** -20,
           flat_pad=2.0):
    """The box test; grid: (o, s), or None for the exact nodes' boxes."""
    with np.errstate(all="ignore"):
        d = b - a
        X = a
        if grid is not None:
            o, s = grid
            X, d = fma32(a - o, s, np.ones_like(a)), d * s
            lo, hi = grid32(lo, hi, o, s)
        ad = np.abs(d)
        flat = ad < F(2.0 ** -62)
        inv = F(1) / d
        inv = np.where(rcp_ulp > 0, np.nextafter(inv, F(np.inf)),
                       np.where(rcp_ulp < 0, np.nextafter(inv, F(-np.inf)), inv)).astype(F)
        i = np.where(flat, F(2.0 ** 62), inv).astype(F)
        c = X * i
        pad = fma32(np.abs(c), np.full_like(c, F(rel)),
                    fma32(np.abs(i), np.full_like(c, F(unit)),
                          np.where(flat, F(flat_pad), F(add)).astype(F)))
        n = -(c + pad)
        f = pad - c
        off = ~((ad <= F(2.0 ** 100)) & (np.abs(c) <= F(2.0 ** 100)))
        i, n, f = (np.where(off, F(v), x).astype(F) for v, x in ((0, i), (-2, n), (2, f)))
        neg = i < 0

        def sat(x):  # NaN clamps to 0
            return np.fmin(np.fmax(x, F(0)), F(1))

        tn = sat(fma32(np.where(neg, hi, lo), i, n)).max(axis=1)
        tf = sat(fma32(np.where(neg, lo, hi), i, f)).min(axis=1)
    return tn < tf


def mesh_box(rng, lo, hi):
    """A mesh box around each box: equal to it, or larger by up to 2^12 box
    sizes, or flat on an axis where the box is."""
    n = lo.shape[0]
    size = (hi.astype(np.float64) - lo).max(axis=1, keepdims=True)
    size = size + np.abs(lo).max(axis=1, keepdims=True) * 1e-6
    grow = size * 2.0 ** rng.uniform(-4, 12, (n, 1)) * rng.choice([0.0, 1.0], (n, 3))
    with np.errstate(all="ignore"):
        mlo = (lo - grow * rng.uniform(0, 1, (n, 3))).astype(F)
        mhi = (hi + grow * rng.uniform(0, 1, (n, 3))).astype(F)
    return np.minimum(mlo, lo), np.maximum(mhi, hi)


def edge_cases(rng):
    """Zero components on a face, ends on a face, far starts, huge and
    infinite differences, and degenerate boxes, as (a, b, lo, hi)."""
    rows = []
    for s in (2.0 ** -90, 2.0 ** -30, 1.0, 2.0 ** 30, 2.0 ** 90, 2.0 ** 126):
        for z in (0.0, 1.0, -1.0):
            a = np.array([z * s, 0.25 * s, -0.5 * s])
            for b in ([z * s, 0.25 * s, 0.5 * s], [z * s, 0.75 * s, -0.5 * s],
                      [z * s + s, 0.25 * s, -0.5 * s], list(a)):
                b = np.array(b)
                for t in (0.0, 0.5, 1.0):
                    x = a + t * (b - a)
                    rows.append((a, b, x, x))
                    rows.append((a, b, x - s * np.array([0, 1, 0]), x + s * np.array([1, 0, 0])))
    return tuple(np.array([r[k] for r in rows]).astype(F) for k in range(4))


def grids(rng, lo, hi):
    return [None, frame32(lo, hi)] + [frame32(*mesh_box(rng, lo, hi)) for _ in range(2)]


@pytest.mark.parametrize("seed", range(3))
def test_touched_boxes_are_never_rejected(seed):
    rng = np.random.default_rng(300 + seed)
    A, B, LO, HI = touching_cases(rng, 20_000)
    for k, grid in enumerate(grids(rng, LO, HI)):
        for ulp in (-1, 0, 1):
            miss = np.nonzero(~walk32(A, B, LO, HI, np.full(A.shape, ulp), grid))[0]
            assert miss.size == 0, (k, ulp, miss[:3])


def test_edge_cases_are_never_rejected():
    rng = np.random.default_rng(0)
    A, B, LO, HI = edge_cases(rng)
    for k, grid in enumerate(grids(rng, LO, HI)):
        for ulp in (-1, 0, 1):
            miss = np.nonzero(~walk32(A, B, LO, HI, np.full(A.shape, ulp), grid))[0]
            assert miss.size == 0, (k, ulp, A[miss[:3]], B[miss[:3]], LO[miss[:3]], HI[miss[:3]])


def test_without_the_pads_touched_boxes_are_lost():
    """A planted mistake: each pad is needed."""
    A, B, LO, HI = touching_cases(np.random.default_rng(300), 20_000)
    up = np.full(A.shape, 1)
    assert (~walk32(A, B, LO, HI, up, rel=0.0, unit=0.0)).sum() > 0
    assert (~walk32(A, B, LO, HI, up, add=0.0)).sum() > 0
    assert (~walk32(A, B, LO, HI, up, unit=0.0, flat_pad=0.0)).sum() > 0


def test_it_rejects_what_the_general_test_rejects():
    """On ordinary boxes the two tests agree (the pads are far below the
    box sizes), and empty boxes are always rejected."""
    rng = np.random.default_rng(5)
    n = 50_000
    a = rng.normal(size=(n, 3)).astype(F)
    b = rng.normal(size=(n, 3)).astype(F)
    lo = rng.normal(size=(n, 3)).astype(F)
    hi = (lo + rng.uniform(0.01, 0.5, size=(n, 3))).astype(F)
    zero = np.zeros((n, 3))
    w, g = walk32(a, b, lo, hi, zero), slab32(a, b, lo, hi, zero)
    assert not (g & ~w).any() and (w != g).mean() < 1e-3
    assert w.any() and not w.all()
    # on a grid 100 box sizes wide the steps are below 1 % of a box
    box = (np.full((n, 3), F(-5)), np.full((n, 3), F(5)))
    q = walk32(a, b, lo, hi, zero, frame32(*box))
    assert not (w & ~q).any() and (w != q).mean() < 1e-3
    # (segments far longer than the mesh may enter them: harmless, the kernel's
    # empty boxes lead to the null triangle)
    gone = walk32(a, b, np.full((n, 3), F(np.inf)), np.full((n, 3), F(-np.inf)), zero,
                  frame32(*box))
    assert not gone.any()
    inf = np.full((n, 3), F(np.inf))
    assert not walk32(a, b, inf, inf, zero).any()
    assert not walk32(a, a, inf, inf, zero).any()
