"""3D steps that rebuild the mixed derivatives, on grids of few blocks (twice the registers, feet
outside the tile both at once) and of more: a COMPACT run against FULL single steps, which read
the stored planes, bit for bit, with feet inside the tiles, at their edge and far outside, on
both sides of the rule (304 blocks of 32 x 4 x 4 nodes)."""
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


# 4, 304, 320 and 390 blocks
@pytest.mark.parametrize("n", [(5, 4, 7), (61, 75, 32), (64, 80, 32), (64, 60, 50)])
@pytest.mark.parametrize("kind", ["const", "rotation", "deform3d"])
@pytest.mark.parametrize("trace", ["rk3", "euler", "heun_psi"])
@pytest.mark.parametrize("cells", [0.5, 1.0, 5.0])
def test_compact_run_equals_full_single_steps(G, n, kind, trace, cells):
    st = inputs.random_state((8,) + tuple(reversed(n)), seed=7, scale=0.3).astype(np.float32)
    vel = G.Velocity(kind, trace=trace, T=3.0, omega=1.0, c=(0.6, -0.8, 0.5))
    dt = cells / (max(n) - 1) / dict(const=0.8, rotation=0.5, deform3d=2.0)[kind]
    a, b = G.Grid(n, layout="compact"), G.Grid(n)
    for g in (a, b):
        g.set_state(st, t0=0.1, recon=True)
    a.step(vel, dt, 3)
    for _ in range(3):
        b.step(vel, dt, 1)
    ra, rb = a.read_state(), b.read_state()
    a.close()
    b.close()
    assert np.array_equal(ra, rb, equal_nan=True)


def test_small_compact_run_with_far_feet_is_no_slower_than_full(G):
    """48^3, a constant field two cells a step: a COMPACT step is one launch where FULL's is two (one
    foot of a thread's two after the other had made it the slower one)."""
    import time

    n = (48, 48, 48)
    st = inputs.sphere_sdf(n, center=(0.45, 0.5, 0.5), r=0.25).astype(np.float32)
    vel, dt = G.Velocity("const", c=(0.6, -0.8, 0.5)), 2.0 / 47 / 0.8

    def best(layout):
        g = G.Grid(n, layout=layout)
        g.set_state(st, recon=True)
        t = []
        for _ in range(12):
            t0 = time.perf_counter()
            g.step(vel, dt, 100)
            g.synchronize()
            t.append(time.perf_counter() - t0)
        g.close()
        return min(t)

    assert best("compact") <= best("full")
