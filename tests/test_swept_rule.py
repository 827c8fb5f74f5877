"""The tile cull's rule: a box is kept iff some t in [0, 1] satisfies six linear
bounds (the swept rectangle from the tile to the target).  Its float32 form,
restated here operation by operation, must never drop a box that meets the
convex hull exactly: integer coordinates on the lattice, with flat, crossing,
touching and far cases in both directions along every axis.
"""

from fractions import Fraction

import numpy as np
import pytest

F = np.float32
U = 1024
PAD = F(0.04)


def kernel_rule(A, B, lo, hi):
    """A, B: (3, 2) float32 low/high of tile and target; lo, hi: box corners."""
    start, stop = F(0), F(1)
    for ax in range(3):
        for a, b, e, upper in ((F(A[ax, 1] + PAD), F(B[ax, 1] + PAD), lo[ax], False),
                               (F(A[ax, 0] - PAD), F(B[ax, 0] - PAD), hi[ax], True)):
            d = F(b - a)
            flat = abs(d) < F(1e-3)
            inv = F(1e30) if flat else F(F(1) / d)
            o = F(F(-a) * inv)
            s = F(np.float64(e) * np.float64(inv) + np.float64(o))   # fused: one rounding (53 bits hold it to < 1e-15)
            if (flat or d > 0) != upper:
                start = max(start, s)
            else:
                stop = min(stop, s)
    return start <= stop


def exact_rule(A, B, lo, hi):
    """The same bounds in rational arithmetic, without the pad."""
    start, stop = Fraction(0), Fraction(1)
    for ax in range(3):
        for a, b, e, upper in ((A[ax, 1], B[ax, 1], lo[ax], False), (A[ax, 0], B[ax, 0], hi[ax], True)):
            a, b, e = (Fraction(int(round(float(x) * U)), U) for x in (a, b, e))
            if b == a:
                if (e > a and not upper) or (e < a and upper):
                    return False
            elif (b > a) != upper:
                start = max(start, (e - a) / (b - a))
            else:
                stop = min(stop, (e - a) / (b - a))
    return start <= stop


@pytest.mark.parametrize("span,grain", [(8, U), (40, 1), (3000, 1), (16384, 1), (16384, U)])
def test_rule_keeps_every_box_that_meets_the_hull(span, grain):
    rng = np.random.default_rng(span + grain)
    met = 0
    for _ in range(1500):
        def pts(width, flat):
            p = rng.integers(-span * U // grain, span * U // grain + 1, 3) * grain
            q = np.minimum(p + rng.integers(0, max(2, width // grain + 1), 3) * grain, 16384 * U)
            q[flat] = p[flat]
            return p, q
        a0, a1 = pts(30 * U, 2)                       # a tile: flat along z
        b0, b1 = pts(40 * U, int(rng.integers(0, 3)))  # a target: flat along its normal
        if rng.random() < 0.3:                        # aligned faces
            k = int(rng.integers(0, 3))
            b1[k] = min(b1[k] - b0[k] + a0[k], 16384 * U)
            b0[k] = a0[k]
        # a box near a point of the hull, often touching it
        t = rng.random()
        mid = ((1 - t) * (a0 + rng.random(3) * (a1 - a0)) + t * (b0 + rng.random(3) * (b1 - b0))).round().astype(np.int64)
        lo = np.clip(mid + rng.integers(-3, 4, 3) * grain * int(rng.integers(0, 20)), -16384 * U, 16384 * U)
        hi = np.minimum(lo + rng.integers(0, 20, 3) * grain, 16384 * U)
        A = np.stack([a0, a1], 1).astype(np.float64) / U
        B = np.stack([b0, b1], 1).astype(np.float64) / U
        l, h = lo / U, hi / U
        exact = exact_rule(A, B, l, h)
        met += exact
        if exact:
            assert kernel_rule(A.astype(F), B.astype(F), l.astype(F), h.astype(F)), (a0, a1, b0, b1, lo, hi)
    assert met > 200
