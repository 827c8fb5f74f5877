"""Direct calls on a stream that is being captured into a CUDA graph: refused in the
modes that do not permit a wait on the host, since the graph would hold scratch
that the context replaces; the context works on afterwards.  No graph is run.
"""

import ctypes

import pytest

import synth
from gpu_util import full_parity

pytestmark = pytest.mark.gpu

GLOBAL, THREAD_LOCAL, RELAXED = 0, 1, 2


@pytest.mark.parametrize("recolor", [False, True])
@pytest.mark.parametrize("mode", [GLOBAL, THREAD_LOCAL, RELAXED])
def test_direct_calls_on_a_capturing_stream(mode, recolor):
    import torch

    import __graft_entry__ as g

    g.build()
    from paper_1310_7297_gb300 import Context, VcmError

    cuda = ctypes.CDLL("libcuda.so.1")
    scene, req = synth.workload_3d(seed=21, grid=24, layers=2, patches=(8, 4), n_boxes=40, half_m=200.0,
                                   n_components=4, sigma_m=(40.0, 90.0))
    with Context(0) as ctx:
        ctx.load_scene(scene)
        ctx.vcm_build(25.0)
        v, c, b, s = ctx.compute(req, emit_bits=True)   # the scratch is allocated
        if recolor:
            ctx.recolor(req, b)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream().cuda_stream
        graph = ctypes.c_void_p()
        assert cuda.cuStreamBeginCapture_v2(ctypes.c_void_p(stream), mode) == 0
        refused = None
        try:
            if recolor:
                ctx.vcm_recolor(req, b.data_ptr(), v.data_ptr(), c.data_ptr(), s.data_ptr(), stream)
            else:
                ctx.vcm_compute(req, v.data_ptr(), c.data_ptr(), None, s.data_ptr(), stream)
        except VcmError as e:
            refused = e
        ended = cuda.cuStreamEndCapture(ctypes.c_void_p(stream), ctypes.byref(graph))
        if graph.value:
            cuda.cuGraphDestroy(graph)
        assert (refused is not None) == (mode != RELAXED)
        assert refused is None or "captur" in str(refused)
        assert (ended == 0) == (mode == RELAXED)
        full_parity(ctx, scene, req)
