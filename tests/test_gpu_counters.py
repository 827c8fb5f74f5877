"""vcm_stats counts work that lanes did: a box tested against a patch column (or
a row group of it) counts once, lanes without a column or without open rows not
at all.
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


@pytest.mark.parametrize("pu,pw", [(1, 1), (20, 1), (45, 13), (3, 11), (32, 16), (2, 5)])
def test_slab_tests_count_the_lanes_with_open_rows(ctx, pu, pw):
    """One box before part of the target: per viewpoint at most one test of each
    column and row group (32 // columns of them, at most one per row)."""
    sc = scene(3, [((-2 * U, 6 * U, 0), (2 * U, 7 * U, 9 * U))])
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req3((0, 0, 8 * U), width=20 * U, height=10 * U, pu=pu, pw=pw, origin=(-10 * U, 12 * U), step=(U, U),
             n=(20, 12), layers=(2 * U, 8 * U))
    _, _, st, _, _ = full_parity(ctx, sc, r)
    groups = min(32 // min(pu, 32), pw)
    assert 0 < st["slab_tests"] <= st["shared_viewpoints"] * pu * groups
