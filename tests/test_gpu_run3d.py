"""3D runs: between the first and the last step of a FULL run the mixed derivatives are rebuilt
around each foot's cell where few feet leave the staged tile, and always in the COMPACT
layout.  A run must equal single steps (stored planes, reconstruction pass) bit for bit:
grids of one tile, a tile and a node, one-sided ends on every side, feet beyond the tile,
both sides of the rule (a reach of 1.05 cells), every velocity and trace."""
import math

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


@pytest.mark.parametrize("n,kind,trace,cells,layout,launches_per_inner_step", [
    ((4, 4, 4), "deform3d", "rk3", 0.5, "full", 1),
    ((33, 5, 9), "rotation", "rk3", 0.9, "full", 1),
    ((32, 40, 24), "deform3d", "rk3", 1.0, "full", 1),
    ((65, 30, 31), "deform3d", "heun_psi", 2.05, "full", 1),   # half of the bound: within the rule
    ((65, 30, 31), "deform3d", "rk3", 2.5, "full", 2),
    ((50, 61, 21), "rotation", "rk3", 1.04, "full", 1),
    ((50, 61, 21), "rotation", "rk3", 1.06, "full", 2),
    ((50, 61, 21), "rotation", "rk3", 4.0, "compact", 1),      # many feet outside the tile
    ((37, 18, 26), "const", "euler", 3.0, "compact", 1),
])
def test_run_equals_single_steps(G, n, kind, trace, cells, layout, launches_per_inner_step):
    st = inputs.random_state((8,) + tuple(reversed(n)), seed=3, scale=0.3).astype(np.float32)
    vel = G.Velocity(kind, trace=trace, T=3.0, omega=2 * math.pi, c=(0.9, -1.0, 0.8))
    bound = {"deform3d": 2.0, "rotation": math.pi, "const": 1.0}[kind]  # the library's speed bounds
    dt = cells / (max(n) - 1) / bound
    a, b = (G.Grid(n, layout=layout) for _ in range(2))
    for g in (a, b):
        g.set_state(st, t0=0.1)
    a.step(vel, dt, 5)
    if layout == "full":  # coefficients, clock, 5 steps, the reconstructions
        assert a.last_step_launches() == 2 + 5 + (1 if launches_per_inner_step == 1 else 5)
    for _ in range(5):
        b.step(vel, dt, 1)
    assert np.array_equal(a.read_state(), b.read_state(), equal_nan=True)
