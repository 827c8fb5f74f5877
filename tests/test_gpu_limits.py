"""Both sides of limits that ordinary requests seldom reach: ids of 3 and 4 bytes
in spill regions and lists too long to publish (the checked build has both limits
at a few hundred boxes), static maps with more open viewpoints than their arena
holds, and viewpoints at the edge of a field of view, where the whole target is
decided at once on one side and patch by patch on the other.
"""

import numpy as np
import pytest

from gpu_util import compare_v, full_parity
from helpers import U, req3, scene
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=["product", "checked"])
def ctx(request):
    import __graft_entry__ as g

    g.build()
    from paper_1310_7297_gb300 import Context

    c = Context(0, checked=request.param == "checked")
    c.is_checked = request.param == "checked"
    yield c
    c.close()


def posts(n, seed):
    """n posts between the viewpoints and the target, all in every list."""
    rng = np.random.default_rng(seed)
    lo = np.stack([rng.integers(-9 * U, 9 * U, n), rng.integers(2 * U, 20 * U, n), np.zeros(n, np.int64)], 1)
    hi = lo + np.stack([rng.integers(30, 500, n), rng.integers(30, 500, n), rng.integers(U, 9 * U, n)], 1)
    return scene(3, list(zip(lo.tolist(), hi.tolist())))


def in_front(**kw):
    return req3((0, 0, 6 * U), width=20 * U, height=8 * U, origin=(-8 * U, 21 * U), step=(U, 2 * U), n=(16, 9),
                layers=(2 * U, 8 * U), **kw)


@pytest.mark.parametrize("n", [64, 299, 301, 333, 599, 601, 902])
def test_spilled_lists(ctx, n):
    """32 boxes staged, the others' ids in spill regions of 3 n or 4 n bytes (n
    where 3 n is not a multiple of 4 among them); past 300 boxes the checked build
    does not publish the list."""
    sc = posts(n, n)
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    ctx.vcm_set_tune(16, 8, 8, 32)
    try:
        _, gb, st, _, _ = full_parity(ctx, sc, in_front(pu=12, pw=7))
    finally:
        ctx.vcm_set_tune(0)
    assert gb.any() and st["error"] == 0 and st["boxes_listed"] > n
    if not ctx.is_checked or n < 300:
        assert st["shared_viewpoints"] > 0
    if ctx.is_checked and n > 500:
        assert st["shared_viewpoints"] < 16 * 9 * 2


@pytest.mark.parametrize("n,pu,pw", [(1100, 4, 2), (1100, 33, 3)])
def test_static_map_past_its_arena(ctx, n, pu, pw):
    """1.2 M viewpoints, nearly all open; the static arena takes half a million and
    the tiles sweep the others."""
    import torch

    from paper_1310_7297_gb300 import stats_from_tensor, vcm

    sc = posts(60, 3)
    r = req3((0, 0, 8 * U), width=6 * U, height=4 * U, pu=pu, pw=pw, origin=(-n // 2 * U, -n // 2 * U), step=(U, U),
             n=(n, n), layers=(90 * U,), flags=8)   # two-sided: the whole grid faces the target
    v = torch.full((n * n,), float("nan"), dtype=torch.float32, device="cuda")
    c = torch.empty(n * n, dtype=torch.uint8, device="cuda")
    s = torch.empty(vcm.STATS_BYTES, dtype=torch.uint8, device="cuda")
    vcm.vcm_compute_static(sc.lo_f32(), sc.hi_f32(), 3, r, v.data_ptr(), c.data_ptr(), None, s.data_ptr(),
                           torch.cuda.current_stream().cuda_stream, checked=ctx.is_checked)
    torch.cuda.synchronize()
    st = stats_from_tensor(s)
    gv = v.cpu().numpy().astype(np.float64)
    assert np.isfinite(gv).all() and st["error"] == 0 and 0 < st["shared_viewpoints"] < (gv > 0).sum()
    idx = np.unique(np.concatenate([np.random.default_rng(1).choice(gv.size, 500), np.arange(0, gv.size, 4093)]))
    compare_v(O.run(sc, r, indices=idx), gv[idx])


@pytest.mark.parametrize("fov,two", [(90.0, 0), (90.0, 8), (120.0, 0), (180.0, 0), (180.0, 8), (270.0, 0)])
@pytest.mark.parametrize("gaze", [(0.0, 1.0, 0.0), (0.5, 1.0, 0.25)])
def test_viewpoints_at_the_edge_of_the_cone(ctx, fov, two, gaze):
    """Viewpoints around the cones of the target's corner patches: for 90 degrees
    along the normal, rows of viewpoints exactly on their edges, and a lattice unit
    to either side of them (2e-5 of the distance, where whole-target decisions give
    way to single patches)."""
    sc = scene(3, [((-U, 9 * U, 0), (U, 10 * U, 9 * U))])
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    # corner patches at x = -7 and 7 m (8 columns 2 m apart), height 8 m (one row)
    for step in (U, U + 1, U - 1):
        r = req3((0, 0, 8 * U), width=16 * U, height=4 * U, pu=8, pw=1, origin=(-30 * U - step // 2, -U // 2),
                 step=(step, U), n=(61, 40), layers=(8 * U, 20 * U), flags=two)
        full_parity(ctx, sc, dict(r, fov_deg=fov, gaze=list(gaze)))
