"""The error word is cleared in the order of the grid's own stream: reported once, whatever the
caller's default stream is busy with, and not cleared late over an error of newer work.  The
checked build's test hook makes a staged-tile wait run out (a child process, GALS_LIB), while
the default stream is kept busy by a kernel of a fraction of a second."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_0905_3409_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

N = (100, 14)  # one block per step


def child():
    import torch

    from paper_0905_3409_gb300 import gals as G
    assert G.LIB_PATH.endswith("libgals_checked.so"), G.LIB_PATH
    torch.zeros(1, device="cuda")
    vel, dt = G.Velocity("vortex2d", T=8.0), 0.9 / (N[0] - 1)
    st = inputs.circle_sdf(N, center=(0.45, 0.55), r=0.3).astype(np.float32)
    assert G.lib().gals_checked_wait_test(2048, 1) == G.OK
    g = G.Grid(N)
    assert G.lib().gals_checked_wait_test(1 << 24, 0) == G.OK
    g.set_state(st, t0=0.2, recon=True)
    out = torch.empty((4, N[1], N[0]), device="cuda")
    torch.cuda.synchronize()

    def outcome(call):
        try:
            call()
            return G.OK
        except G.GalsError as e:
            return e.status

    def read():
        ptrs = (G.ctypes.c_void_p * 4)(*[out[p].data_ptr() for p in range(4)])
        G._check(G.lib().gals_read_state(g._h, ptrs, 4, G.MEM_DEVICE), g._h)

    got = []
    for call in (g.synchronize, read):
        g.step(vel, dt, 1)
        torch.cuda._sleep(800_000_000)          # the default stream, about 0.4 s
        got += [outcome(call), outcome(call)]   # reported, then clear
        g.step(vel, dt, 1)
        torch.cuda.synchronize()                # whatever is queued anywhere has run
        got += [outcome(call), outcome(call)]   # the newer error is reported too
    print(got)
    assert got == [G.ERR_TIMEOUT, G.OK] * 4, got
    g.close()


def test_error_word_is_reported_once_on_a_busy_default_stream():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0905_3409_gb300 import build
    env = dict(os.environ, GALS_LIB=build.build_checked())
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]


if __name__ == "__main__":
    child()
