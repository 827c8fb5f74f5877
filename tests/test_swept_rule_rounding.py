"""The tile cull's rule with the hardware's reciprocal: the kernel's 1/d is up to
one unit in the last place from the rounded quotient.  With every reciprocal moved
by one unit either way the rule must still keep each box that meets the hull.
"""

import numpy as np
import pytest

from test_swept_rule import PAD, U, exact_rule

F = np.float32


def rule(A, B, lo, hi, move):
    """The kernel's rule; move[k] in {-1, 0, 1}: units added to the k-th 1/d."""
    start, stop, k = F(0), F(1), 0
    for ax in range(3):
        for a, b, e, upper in ((F(A[ax, 1] + PAD), F(B[ax, 1] + PAD), lo[ax], False),
                               (F(A[ax, 0] - PAD), F(B[ax, 0] - PAD), hi[ax], True)):
            d = F(b - a)
            flat = abs(d) < F(1e-3)
            inv = F(1e30) if flat else F(F(1) / d)
            if not flat and move[k]:
                inv = np.nextafter(inv, F(np.inf) if move[k] > 0 else F(-np.inf))
            k += 1
            s = F(np.float64(e) * np.float64(inv) + np.float64(F(F(-a) * inv)))
            if (flat or d > 0) != upper:
                start = max(start, s)
            else:
                stop = min(stop, s)
    return start <= stop


@pytest.mark.parametrize("span,grain", [(8, U), (3000, 1), (16384, 1), (16384, U)])
def test_rule_holds_with_reciprocals_a_unit_off(span, grain):
    rng = np.random.default_rng(span * 7 + grain)
    met = 0
    for _ in range(800):
        a0 = rng.integers(-span * U // grain, span * U // grain + 1, 3) * grain
        a1 = np.minimum(a0 + rng.integers(0, 30 * U // grain + 1, 3) * grain, 16384 * U)
        b0 = rng.integers(-span * U // grain, span * U // grain + 1, 3) * grain
        b1 = np.minimum(b0 + rng.integers(0, 40 * U // grain + 1, 3) * grain, 16384 * U)
        a1[2] = a0[2]
        flat = int(rng.integers(0, 2))
        b1[flat] = b0[flat]
        t = rng.random()
        # a corner of the box at a vertex of the hull's section, so that many only touch it
        side_a, side_b = np.where(rng.random(3) < 0.5, a0, a1), np.where(rng.random(3) < 0.5, b0, b1)
        at = ((1 - t) * side_a + t * side_b).round().astype(np.int64)
        size = rng.integers(0, 20, 3) * grain
        lo = np.where(rng.random(3) < 0.5, at, at - size)
        lo, hi = np.clip(lo, -16384 * U, 16384 * U), np.clip(lo + size, -16384 * U, 16384 * U)
        A, B = np.stack([a0, a1], 1).astype(np.float64) / U, np.stack([b0, b1], 1).astype(np.float64) / U
        l, h = lo / U, hi / U
        if not exact_rule(A, B, l, h):
            continue
        met += 1
        for move in ([1] * 6, [-1] * 6, rng.integers(-1, 2, 6)):
            assert rule(A.astype(F), B.astype(F), l.astype(F), h.astype(F), move), (a0, a1, b0, b1, lo, hi, move)
    assert met > 200
