"""make_request packs a request in one go; the result must be the struct that
assigning its fields one by one gives, for plain, numpy and out-of-range values.
"""

import math

import numpy as np
import pytest

import synth
from paper_1310_7297_gb300 import vcm


def fields(r):
    out = []
    for name, _ in vcm.vcm_request._fields_:
        x = getattr(r, name)
        if name == "layer_z":
            x = [x[i] for i in range(r.n_layers)]
        out.append(list(x) if hasattr(x, "__len__") else [x])
    return out


@pytest.mark.parametrize("change", [
    {}, {"fov_deg": 120.0, "gaze": (0.5, -0.25, 1e-3), "v_ref": 0.1, "flags": 9}, {"layer_z": np.array([1, 2, 3])},
    {"center": np.array([5, -7, 11])}, {"layer_z": []}, {"grid_nx": -1}, {"width": float("nan")}, {"height": 10 ** 45},
    {"v_ref": 1e300}, {"layer_z": [1.5, float("inf")]}, {"gaze": np.array([1.0, 2.0, 3.0])}])
def test_packed_request_equals_field_by_field(change):
    req = dict(synth.workload_3d(n_boxes=3)[1], **change)
    a, keep_a = vcm.make_request(req)
    b, keep_b = vcm._make_request_by_field(req)
    for x, y in zip(fields(a), fields(b)):
        assert len(x) == len(y) and all(p == q or (math.isnan(p) and math.isnan(q)) for p, q in zip(x, y))


def test_wrong_types_are_refused():
    req = synth.workload_3d(n_boxes=3)[1]
    for change in ({"grid_nx": 2.5}, {"dims": "3"}, {"width": None}):
        with pytest.raises(TypeError):
            vcm.make_request(dict(req, **change))
