"""Batched problems of the vortex and rotation fields, in FULL and COMPACT runs, evolve bit for bit
as on their own grids, for both tile heights, one block per tile and persistent blocks, runs of
one, two and four steps."""
import numpy as np
import pytest

from paper_0905_3409_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [(130, 97), (37, 41), (128, 129), (300, 17), (5, 4), (129, 16)]


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    from paper_0905_3409_gb300 import gals
    return gals


@pytest.mark.parametrize("layout", ["full", "compact"])
@pytest.mark.parametrize("kind,cells", [("vortex2d", 0.9), ("rotation", 0.9), ("rotation", 3.0)])
def test_batch_equals_single_grids(G, layout, kind, cells):
    vel = G.Velocity(kind, T=8.0, omega=2.0)
    states = [inputs.circle_sdf(n, center=(0.45, 0.55), r=0.3).astype(np.float32) for n in SIZES]
    dts = [cells / (max(n) - 1) for n in SIZES]
    want = []
    for n, st, dt in zip(SIZES, states, dts):
        g = G.Grid(n, layout=layout)
        g.set_state(st, t0=0.2, recon=True)
        for _ in range(7):
            g.step(vel, dt, 1)
        want.append(g.read_state())
        g.close()
    for variant, blocks in ((0, 0), (1, 0), (0, 5), (1, 3)):
        b = G.Batch(SIZES, layout=layout)
        for p, st in enumerate(states):
            b.set_state(p, st, t0=0.2, recon=True)
        b.set_tuning(variant, blocks)
        for steps in (1, 2, 4):
            b.step([vel] * len(SIZES), dts, steps)
        for p, w in enumerate(want):
            assert np.array_equal(b.read_state(p), w), (variant, blocks, p)
        b.close()
