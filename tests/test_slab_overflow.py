"""CPU check of the general loop's segment / box test where a segment's
difference overflows (csrc/rsi_internal.cuh, slab_rcp): its reciprocal is NaN
there, and the test's minima and maxima drop the axis, so no box that the exact
segment touches is rejected; with the reciprocal 0 they are.  And why an empty
slot needs a leaf that is safe to test: with all three axes dropped its box
(+inf) is entered too."""
from fractions import Fraction

import numpy as np

F = np.float32
SLACK = F(1 + 2.0 ** -18)


def slab(a, b, lo, hi, inf_rcp):
    with np.errstate(all="ignore"):
        d = b - a
        inv = np.where(np.isinf(d), F(inf_rcp), F(1) / d).astype(F)
        neg = inv < 0
        tn = (np.where(neg, hi, lo) - a) * inv
        tf = (np.where(neg, lo, hi) - a) * inv
        tn = np.fmax(np.fmax(tn[:, 0], tn[:, 1]), np.fmax(tn[:, 2], F(0)))
        tf = np.fmin(np.fmin(tf[:, 0], tf[:, 1]), np.fmin(tf[:, 2], F(1)))
        return tn <= tf * SLACK


def cases(n=4000):
    """Segments with finite ends and at least one overflowing difference, and
    boxes around a point of each that is known exactly."""
    rng = np.random.default_rng(12)
    A, B, LO, HI = (np.empty((n, 3), F) for _ in range(4))
    for i in range(n):
        a = (rng.uniform(-1, 1, 3) * 3.4e38).astype(F)
        b = (rng.uniform(-1, 1, 3) * 3.4e38).astype(F)
        for k in rng.choice(3, rng.integers(1, 4), replace=False):
            a[k], b[k] = F(rng.uniform(-3.4e38, -2e38)), F(rng.uniform(2e38, 3.4e38))
            if rng.integers(2):
                a[k], b[k] = b[k], a[k]
        s = Fraction(int(rng.integers(0, 1025)), 1024)
        for k in range(3):
            x = Fraction(float(a[k])) + s * (Fraction(float(b[k])) - Fraction(float(a[k])))
            f = F(float(x))
            LO[i, k] = np.nextafter(f, F(-np.inf)) if Fraction(float(f)) > x else f
            HI[i, k] = np.nextafter(f, F(np.inf)) if Fraction(float(f)) < x else f
        A[i], B[i] = a, b
    return A, B, LO, HI


def test_touched_boxes_are_never_rejected():
    A, B, LO, HI = cases()
    with np.errstate(all="ignore"):
        assert np.isinf(B - A).any(axis=1).all()
    assert slab(A, B, LO, HI, np.nan).all()


def test_with_a_zero_reciprocal_they_are():
    assert (~slab(*cases(), 0.0)).sum() > 100


def test_an_empty_slot_is_entered_by_a_segment_that_overflows_everywhere():
    A, B, LO, HI = cases()
    with np.errstate(all="ignore"):
        every = np.isinf(B - A).all(axis=1)
    inf = np.full_like(LO, np.inf)
    got = slab(A, B, inf, inf, np.nan)
    assert every.any() and np.array_equal(got, every)
