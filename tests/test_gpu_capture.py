"""gals_step on a stream that its caller is capturing: a call of several steps, which launches
cached graphs or the small grids' cluster run and moves the host's clock, is refused, on a
small grid as on a larger one, and leaves the grid as it was; the same call after the
capture steps as on a grid that was never captured."""
import ctypes

import numpy as np
import pytest

from paper_0905_3409_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    from paper_0905_3409_gb300 import gals
    return gals


@pytest.mark.parametrize("n,steps", [((64, 64), 8), ((64, 64), 9), ((64, 64), 300), ((64, 64), 7), ((300, 200), 8)])
def test_several_steps_are_refused_while_captured(G, n, steps):
    import torch

    vel, dt = G.Velocity("vortex2d", T=8.0), 0.8 / (max(n) - 1)
    st = inputs.circle_sdf(n).astype(np.float32)
    stream = torch.cuda.Stream()
    a, b = G.Grid(n, stream=stream), G.Grid(n)
    for g in (a, b):
        g.set_state(st, t0=0.2, recon=True)
        g.step(vel, dt, steps)          # tables and attributes are there before the capture
        g.synchronize()
    t, launches = a.time, a.last_step_launches()
    # by the runtime itself: a capture that the refused call ends early would leave torch's
    # allocator waiting for the end of it
    rt, graph, s = ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p(), ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(s, ctypes.c_int(1)) == 0  # thread-local mode
    try:
        with pytest.raises(G.GalsError) as e:
            a.step(vel, dt, steps)
    finally:
        rt.cudaStreamEndCapture(s, ctypes.byref(graph))
        if graph:
            rt.cudaGraphDestroy(graph)
        rt.cudaGetLastError()
    assert e.value.status == G.ERR_CUDA
    assert a.time == t
    assert np.array_equal(a.read_state(), b.read_state())
    for g in (a, b):
        g.step(vel, dt, steps)
    assert a.last_step_launches() == launches
    assert np.array_equal(a.read_state(), b.read_state())
