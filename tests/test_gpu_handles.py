"""Creating and destroying handles: the page-locked word that a handle reads its error word from
is shared out of a slab, so that a small grid's life costs less than one page-locked
allocation (with an allocation of its own it cost three and a half times what it had); more
handles than a slab has words, from several threads, given back in any order, each keep
their own word."""
import ctypes
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_0905_3409_gb300 import inputs  # noqa: E402

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


def _best(call, reps=30):
    t = []
    for _ in range(reps):
        t0 = time.perf_counter()
        call()
        t.append(time.perf_counter() - t0)
    return min(t)


def child():
    """In a process of its own: page-locked allocations are cheap while another one is alive."""
    import torch
    from paper_0905_3409_gb300 import gals as G

    torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    rt, p = ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p()

    def page_locked():
        assert rt.cudaMallocHost(ctypes.byref(p), ctypes.c_size_t(4)) == 0
        assert rt.cudaFreeHost(p) == 0

    alone = _best(page_locked)
    grid = _best(lambda: G.Grid((64, 64)).close())
    print(f"page-locked word {alone * 1e6:.0f} us, grid {grid * 1e6:.0f} us")
    assert grid <= alone


def test_a_small_grid_costs_less_than_a_page_locked_allocation(G):
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]


def test_many_handles_from_several_threads(G):
    vel, n = G.Velocity("vortex2d", T=8.0), (6, 5)
    st = inputs.circle_sdf(n).astype(np.float32)
    want = G.Grid(n)
    want.set_state(st, recon=True)
    want.step(vel, 0.1, 1)
    ref = want.read_state()
    bad = []

    def life(seed):
        try:
            rng = np.random.default_rng(seed)
            held = []
            for _ in range(600):
                g = G.Grid(n)
                g.set_state(st, recon=True)
                held.append(g)
                if len(held) > 400 or rng.random() < 0.2:
                    g = held.pop(rng.integers(len(held)))
                    g.step(vel, 0.1, 1)
                    if not np.array_equal(g.read_state(), ref):
                        bad.append(seed)
                    g.close()
            for g in held:
                g.synchronize()
                g.close()
        except Exception as e:  # noqa: BLE001
            bad.append(e)

    threads = [threading.Thread(target=life, args=(s,)) for s in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[:3]


if __name__ == "__main__":
    child()
