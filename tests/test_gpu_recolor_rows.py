"""Recolouring of targets with more patch rows than 256, and with one or the most
there can be: the values equal the oracle's within 1e-5, as everywhere, with the
side, the cone and strictness applied to bits made without them.
"""

import numpy as np
import pytest

from gpu_util import compare_v
from helpers import U, req3, scene
from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g

    g.build()
    from paper_1310_7297_gb300 import Context

    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("pu,pw", [(7, 300), (32, 300), (3, 4096), (1, 257), (4096, 1), (33, 256)])
def test_recolor_with_many_rows(ctx, pu, pw):
    import torch

    sc = scene(3, [((-3 * U, 5 * U, 0), (2 * U, 6 * U, 7 * U)), ((-9 * U, 7 * U, 0), (-6 * U, 9 * U, 14 * U))])
    ctx.load_scene(sc)
    ctx.vcm_build(0.0)
    r = req3((0, 0, 8 * U), width=14 * U, height=12 * U, pu=pu, pw=pw, origin=(-12 * U, -6 * U), step=(2 * U, 3 * U),
             n=(11, 9), layers=(2 * U, 9 * U))
    bits = ctx.compute(r, emit_bits=True)[2]
    for change in ({}, {"flags": 8, "fov_deg": 120.0, "gaze": [0.25, 1.0, -0.125]}, {"fov_deg": 330.0}, {"flags": 2}):
        q = dict(r, **change)
        v = ctx.recolor(q, bits)[0]
        torch.cuda.synchronize()
        ov, band = O.run(sc, q, band=True)
        compare_v(ov, v.cpu().numpy().astype(np.float64), str(change), band)
