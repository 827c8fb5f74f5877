"""The tile cull on the device: boxes that touch the hull of a tile and the target
in a point, an edge or a face, near and 16 km out, must not be dropped.  A
touching box blocks the segment it touches, so the bits show it.
"""

import numpy as np
import pytest

from gpu_util import full_parity
from helpers import U, req3, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g

    g.build()
    from paper_1310_7297_gb300 import Context

    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("far", [0, 1, 2], ids=["near", "3km", "16km"])
@pytest.mark.parametrize("axis_u,axis_w,normal", [(0, 4, 2), (3, 4, 0), (0, 2, 4)])
def test_touching_boxes_are_kept(ctx, axis_u, axis_w, normal, far):
    """One tile of 8 x 4 viewpoints; each box has a corner on the middle of a
    segment from an extreme viewpoint to an extreme patch (even coordinates, so
    that the middle is on the lattice) and lies outside the hull but for that."""
    rng = np.random.default_rng(100 * far + 10 * axis_u + normal)
    base = (0, 2800 * U, 15900 * U)[far]
    lim = 16384 * U
    n_axis, u_axis, w_axis = normal >> 1, axis_u >> 1, axis_w >> 1
    sign = -1 if normal & 1 else 1
    blocked = 0
    for trial in range(12):
        # the target's far corner and the tile, apart along the normal; whole pairs of units
        centre = [0, 0, 0]
        centre[u_axis] = int(rng.integers(-200, 200)) * 2 * U + (base if far else 0) * (1 if trial % 2 else -1)
        centre[w_axis] = int(rng.integers(0, 40)) * 2 * U
        origin = [int(rng.integers(-100, 100)) * 2 * U, int(rng.integers(-100, 100)) * 2 * U]
        z = int(rng.integers(0, 60)) * 2 * U
        if n_axis < 2:
            origin[n_axis] = sign * int(rng.integers(60, 200)) * U - (0 if sign > 0 else 4 * 4 * U)
        else:
            z = sign * int(rng.integers(60, 200)) * 2 * U
            centre[n_axis] = 0
        centre = [int(np.clip(x, -lim + 60 * U, lim - 60 * U)) for x in centre]
        # patch centres at +-6 m and +-2 m around the centre: 8 m and 4 m steps of 4 columns, 2 rows
        r = req3(centre, axis_u=axis_u, axis_w=axis_w, normal=normal, width=16 * U, height=8 * U, pu=4, pw=2,
                 origin=origin, step=(4 * U, 4 * U), n=(8, 4), layers=(z,))
        p = np.array(centre)
        su, sw = rng.choice([-1, 1]), rng.choice([-1, 1])
        p[u_axis] += su * 6 * U
        p[w_axis] += sw * 2 * U
        ix, iy = int(rng.choice([0, 7])), int(rng.choice([0, 3]))
        q = np.array([origin[0] + 4 * U * ix + 2 * U, origin[1] + 4 * U * iy + 2 * U, z])
        mid = (p + q) // 2
        out = np.where(q + p - np.array([2 * origin[0] + 32 * U, 2 * origin[1] + 16 * U, 2 * z]) >= 0, 1, -1)
        size = rng.integers(0, 3, 3) * U
        lo, hi = np.minimum(mid, mid + out * size), np.maximum(mid, mid + out * size)
        # not on the target itself
        keep = np.abs(mid - np.array(centre)).max() > 30 * U
        if not keep:
            continue
        lo, hi = np.clip(lo, -lim, lim), np.clip(hi, -lim, lim)
        sc = scene(3, [(lo.tolist(), hi.tolist())])
        ctx.load_scene(sc)
        ctx.vcm_build(0.0)
        ctx.vcm_set_tune(8, 4, 8, 32)
        try:
            _, gb, _, _, _ = full_parity(ctx, sc, r)
        finally:
            ctx.vcm_set_tune(0)
        blocked += int(gb.any())
    assert blocked >= 6
