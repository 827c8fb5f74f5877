"""The sweep's row intervals (one bit mask of up to 32 rows per lane) where
they can go wrong: more rows than a mask holds, a last group of one row, rows
running down the w axis, rows so close together that they round to the same
lattice heights, viewpoints far enough that a row number loses its fraction,
and box faces on row heights and patch columns.  Bits must equal the oracle's
exactly and values lie within 1e-5, as everywhere.
"""

import numpy as np
import pytest

from gpu_util import full_parity
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


def field(seed, centre, keep=(7, 2, 5)):
    """90 boxes on whole metres, none within `keep` metres of `centre`."""
    rng = np.random.default_rng(seed)
    lo = rng.integers(-60, 60, size=(90, 3)) * U
    lo[:, 2] = rng.integers(0, 12, size=90) * U
    hi = lo + rng.integers(1, 9, size=(90, 3)) * U
    keep = np.array(keep) * U
    off = ~np.all((lo <= np.asarray(centre) + keep) & (np.asarray(centre) - keep <= hi), axis=1)
    return scene(3, list(zip(lo[off].tolist(), hi[off].tolist())))


@pytest.mark.parametrize("pu,pw", [(1, 1), (2, 33), (32, 31), (32, 33), (33, 65), (5, 200), (31, 64), (64, 40),
                                   (3, 11), (100, 3)])
def test_rows_per_mask(ctx, pu, pw):
    c = (0, 0, 8 * U)
    sc = field(pu * 1000 + pw, c)
    ctx.load_scene(sc)
    ctx.vcm_build(10.0)
    r = req3(c, width=12 * U, height=8 * U, pu=pu, pw=pw, origin=(-50 * U, -50 * U), step=(7 * U, 9 * U), n=(14, 11),
             layers=(2 * U, 8 * U))
    _, gb, st, _, _ = full_parity(ctx, sc, r)
    assert gb.any() and st["slab_tests"] > 0


@pytest.mark.parametrize("axis_u,axis_w,normal", [(0, 5, 2), (1, 4, 3), (2, 5, 1), (0, 3, 4), (4, 1, 2)])
def test_descending_rows_and_other_frames(ctx, axis_u, axis_w, normal):
    c = (0, 0, 14 * U)
    sc = field(axis_u + 10 * axis_w, c, (8, 8, 8))
    ctx.load_scene(sc)
    ctx.vcm_build(10.0)
    r = req3(c, axis_u=axis_u, axis_w=axis_w, normal=normal, width=10 * U, height=10 * U, pu=20, pw=20,
             origin=(-45 * U, -45 * U), step=(6 * U, 6 * U), n=(15, 15), layers=(3 * U, 14 * U, 25 * U))
    full_parity(ctx, sc, r)


@pytest.mark.parametrize("height,pw,far", [(1, 4, 0), (20, 64, 0), (700, 48, 0), (3 * U, 40, 15000), (8 * U, 64, 15000)])
def test_rows_closer_than_a_row_number_resolves(ctx, height, pw, far):
    """Rows of a few lattice units (or all equal), and targets whose rows lie
    0.07-0.12 m apart seen from layers far above them."""
    c = (0, 0, 8 * U)
    sc = field(height + pw, c)
    ctx.load_scene(sc)
    ctx.vcm_build(10.0)
    layers = (8 * U, far * U) if far else (7 * U, 8 * U, 9 * U)
    r = req3(c, width=12 * U, height=height, pu=16, pw=pw, origin=(-50 * U, -50 * U), step=(9 * U, 9 * U),
             n=(11, 11), layers=layers)
    full_parity(ctx, sc, r)


def test_faces_on_rows_and_columns(ctx):
    """Rows and columns on whole metres, as the boxes' faces: both ends of
    many intervals fall on a row."""
    c = (0, 0, 16 * U)
    sc = field(5, c, (17, 2, 17))
    ctx.load_scene(sc)
    ctx.vcm_build(10.0)
    r = req3(c, width=32 * U, height=32 * U, pu=16, pw=16, origin=(-49 * U, -49 * U), step=(2 * U, 2 * U), n=(49, 49),
             layers=(1 * U, 5 * U, 9 * U))
    _, _, st, _, _ = full_parity(ctx, sc, r)
    assert st["rechecked"] > 0


@pytest.mark.parametrize("pu", [1, 31, 33, 70])
def test_2d_columns(ctx, pu):
    rng = np.random.default_rng(pu)
    lo = rng.integers(-40, 40, size=(60, 3)) * U
    hi = lo + rng.integers(1, 6, size=(60, 3)) * U
    lo[:, 2] = hi[:, 2] = 0
    off = ~np.all((lo[:, :2] <= np.array([9, 1]) * U) & (np.array([-9, -1]) * U <= hi[:, :2]), axis=1)
    sc = scene(2, list(zip(lo[off].tolist(), hi[off].tolist())))
    ctx.load_scene(sc)
    ctx.vcm_build(8.0)
    full_parity(ctx, sc, req2((0, 0), width=16 * U, pu=pu, origin=(-40 * U, -40 * U), step=(2 * U, 2 * U), n=(40, 40)))


def test_more_boxes_per_viewpoint_than_records(ctx):
    """300 posts between the viewpoints and the target: more boxes left to a
    viewpoint than it keeps records for (32), and longer lists than a warp
    stages (64)."""
    posts = []
    for i in range(60):
        for j in range(5):
            x, y = (i - 30) * U // 2 + 100 * j, (4 + 2 * j) * U
            posts.append(((x, y, 0), (x + 77, y + 90, (6 + (i * 7 + j * 3) % 9) * U)))
    sc = scene(3, posts)
    ctx.load_scene(sc)
    ctx.vcm_build(4.0)
    r = req3((0, 0, 8 * U), width=20 * U, height=10 * U, pu=64, pw=40, origin=(-12 * U, 14 * U), step=(U, 2 * U),
             n=(24, 12), layers=(2 * U, 9 * U))
    _, gb, _, _, _ = full_parity(ctx, sc, r)
    assert gb.any()


@pytest.mark.parametrize("n", (4096, 7232), ids=("one-round", "rounds"))
def test_more_open_viewpoints_than_the_arena_holds(ctx, n):
    """Nearly all viewpoints open, and more of them than the second pass's arena
    (12.8 M) takes: the tiles sweep the rest of 16.8 M, 52.3 M run in rounds."""
    from gpu_util import compare_bits, compare_v, gpu_run
    from oracle import oracle as O

    sc = field(77, (0, 0, 8 * U))
    ctx.load_scene(sc)
    ctx.vcm_build(10.0)
    r = req3((0, 0, 8 * U), width=6 * U, height=4 * U, pu=4, pw=2, origin=(-n // 2 * U, -n // 2 * U), step=(U, U),
             n=(n, n), layers=(300 * U,), flags=8)   # two-sided: the whole grid faces the target
    gv, _, gb, st = gpu_run(ctx, r, bits=True)
    assert np.isfinite(gv).all() and 0 < st["shared_viewpoints"] < gv.size
    assert n == 4096 or st["shared_viewpoints"] > 13000000
    idx = np.unique(np.concatenate([np.random.default_rng(1).choice(gv.size, 600), np.arange(0, gv.size, 65521)]))
    ov, ob = O.run(sc, r, indices=idx, bits=True)
    compare_bits(ob, gb[idx])
    compare_v(ov, gv[idx])
