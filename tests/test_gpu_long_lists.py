"""Viewpoints with candidate lists of hundreds of boxes: the sweep takes the
nearest ones first and stops when no patch is left open, and the results equal
the oracle's for every patch grid, mode and list length around its limits (256
boxes, the 448 that a tile stages).
"""

import numpy as np
import pytest

from gpu_util import full_parity, gpu_run
from helpers import U, req2, req3, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g

    g.build()
    from paper_1310_7297_gb300 import Context

    c = Context(0)
    yield c
    c.close()


def walled(n):
    """Two walls beside each other, 4 m in front of the viewpoints, neither of
    which hides the whole target, and n posts just in front of the target."""
    boxes = [((-60 * U, 36 * U, 0), (0, 37 * U, 40 * U)), ((0, 36 * U, 0), (60 * U, 37 * U, 40 * U))]
    for i in range(n):
        x = -10 * U + (i % 100) * U // 5
        y = 2 * U + (i // 100) * U
        boxes.append(((x, y, 0), (x + 90, y + 200, (3 + i % 11) * U)))
    return scene(3, boxes)


@pytest.mark.parametrize("flags", [0, 2], ids=["plain", "strict"])
def test_near_boxes_end_a_long_list(ctx, flags):
    """Every viewpoint is hidden by one or both of the two nearest boxes of about
    400.  The counters show that the others are not looked at: at most 48 box tests
    per viewpoint are the tile's own checks, and a viewpoint that needs both walls
    takes the 32 boxes of the first step."""
    sc = walled(400)
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req3((0, 0, 8 * U), width=20 * U, height=10 * U, pu=32, pw=16, origin=(-3 * U, 41 * U), step=(U // 4, U // 4),
             n=(24, 24), layers=(4 * U, 8 * U), flags=flags)
    gv, gb, st, _, _ = full_parity(ctx, sc, r, bits=False)
    assert not gv.any() and st["shared_viewpoints"] > 500
    tiles = -(-24 // 8) * -(-24 // 4) * 2   # at most: tiles of 8 x 4
    assert st["boxes_listed"] > 300 * 8 and st["boxes_listed"] <= 402 * tiles
    assert st["corner_tests"] // 4 + st["slab_tests"] // 32 <= 48 * gv.size + 32 * st["shared_viewpoints"]


@pytest.mark.parametrize("n", [250, 258, 447, 1300])
@pytest.mark.parametrize("pu,pw,flags", [(8, 4, 0), (33, 40, 0), (64, 40, 8), (32, 16, 2), (1, 70, 10)])
def test_long_lists_equal_the_oracle(ctx, n, pu, pw, flags):
    rng = np.random.default_rng(n + pu)
    lo = np.stack([rng.integers(-24 * U, 24 * U, n), rng.integers(2 * U, 30 * U, n), np.zeros(n, np.int64)], 1)
    hi = lo + np.stack([rng.integers(30, 900, n), rng.integers(30, 900, n), rng.integers(U, 14 * U, n)], 1)
    hi[::17, 0] += 12 * U   # some of them hide much of the target
    sc = scene(3, list(zip(lo.tolist(), hi.tolist())))
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req3((0, 0, 6 * U), width=24 * U, height=9 * U, pu=pu, pw=pw, origin=(-20 * U, 5 * U), step=(3 * U, 3 * U),
             n=(13, 13), layers=(2 * U, 9 * U), flags=flags)
    full_parity(ctx, sc, r)
    full_parity(ctx, sc, r, bits=False)


@pytest.mark.parametrize("pu", [8, 70])
def test_long_lists_in_2d(ctx, pu):
    rng = np.random.default_rng(pu)
    lo = np.stack([rng.integers(-40 * U, 40 * U, 1500), rng.integers(2 * U, 50 * U, 1500), np.zeros(1500, np.int64)], 1)
    hi = lo + np.stack([rng.integers(10, 700, 1500), rng.integers(10, 700, 1500), np.zeros(1500, np.int64)], 1)
    sc = scene(2, list(zip(lo.tolist(), hi.tolist())))
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req2((0, 0), width=40 * U, pu=pu, origin=(-32 * U, 3 * U), step=(2 * U, 2 * U), n=(32, 24))
    for flags in (0, 2):
        full_parity(ctx, sc, dict(r, flags=flags))
    gv, _, _, st = gpu_run(ctx, r, bits=False)
    assert st["error"] == 0 and st["boxes_listed"] > 0


@pytest.mark.parametrize("n", [1, 31, 32, 33, 34, 63, 64, 65, 98])
@pytest.mark.parametrize("wall", [False, True], ids=["posts", "wall"])
@pytest.mark.parametrize("pu,pw,flags", [(40, 40, 0), (16, 8, 2), (3, 70, 8)])
def test_kept_boxes_around_the_records_that_a_viewpoint_holds(ctx, n, wall, pu, pw, flags):
    """Up to n posts in a viewpoint's view (32 records are held; with more the passes
    filter the list), without and with a box behind them that hides the whole
    target."""
    boxes = [((-9 * U + i * 18 * U // n, 8 * U + i * U // 8, 0), (-9 * U + i * 18 * U // n + 60, 8 * U + i * U // 8 + 60, 9 * U))
             for i in range(n)]
    if wall:
        boxes.append(((-30 * U, 2 * U, 0), (30 * U, 3 * U, 40 * U)))
    sc = scene(3, boxes)
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req3((0, 0, 6 * U), width=24 * U, height=9 * U, pu=pu, pw=pw, origin=(-4 * U, 24 * U), step=(U, 2 * U),
             n=(9, 7), layers=(2 * U, 8 * U), flags=flags)
    gv, _, st, _, _ = full_parity(ctx, sc, r, bits=False)
    full_parity(ctx, sc, r)
    assert st["error"] == 0 and (not wall or not gv.any())
