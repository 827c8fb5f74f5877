"""Boxes that graze segments, in few columns (their rows are spread over the lanes)
and in all of them (every lane decides its own): viewpoints in the planes of box
faces and targets whose patches lie on them.  Bits must equal the oracle's.
"""

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


@pytest.mark.parametrize("pu,pw", [(28, 8), (4, 22), (1, 32), (2, 64), (33, 33), (8, 4), (64, 3)])
def test_grazing_rows(ctx, pu, pw):
    """Viewpoints at x = 0 .. 15 m and heights 0, 4 and 8 m: box faces lie in their
    planes, so whole columns (a face at the viewpoint's x) or every column (a face
    in the plane of the target's normal through it) graze."""
    boxes = []
    for i in range(16):
        x, y = i * U, (4 + i % 3) * U
        boxes.append(((x, y, 0), (x + U, y + U // 2, (4 + 4 * (i % 2)) * U)))
        boxes.append(((x - 9 * U, (8 + i) * U, 0), (x + 9 * U, (9 + i) * U, (1 + i % 4) * U)))
    sc = scene(3, boxes)
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req3((8 * U, 0, 4 * U), width=pu * U // 2, height=8 * U, pu=pu, pw=pw, origin=(-U // 2, 7 * U + U // 2),
             step=(U, U), n=(16, 18), layers=(0, 4 * U, 8 * U))
    for flags in (0, 2):
        _, gb, st, _, _ = full_parity(ctx, sc, dict(r, flags=flags))
        assert gb.any() and st["rechecked"] > 0
