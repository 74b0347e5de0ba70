"""Fields of 64 and more plane waves, whose steps take 2-row tiles as far as a launch holds them
(65535 tiles along y, 131070 rows) and 14-row tiles on taller grids: strips on both sides of
that line, at the most rows a grid may have and on a size whose four bands are each within
the line while the whole grid is not; and a grid of more than 850 tall tiles, where other
fields' steps are tall.  Single steps against the FP64 oracle (max |dphi| <= 1e-5,
max |dpsi| <= 1e-4), runs against single steps bit for bit."""
import numpy as np
import pytest

import oracle
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


def _strip(rows):
    h = 1.0 / (rows - 1)
    lo, hi = (0.3, 0.0), (0.3 + 4 * h, 1.0)                 # square cells
    st = inputs.circle_sdf((5, rows), center=(0.3, 0.5), r=0.2, lo=lo, hi=hi).astype(np.float32)
    return h, lo, hi, st


@pytest.mark.parametrize("rows", [131070, 131071, 917490])
def test_strip_step_against_oracle(G, rows):
    modes = inputs.wave_modes(64, seed=17)
    h, lo, hi, st = _strip(rows)
    dt = 0.8 * h / inputs.wave_speed_sampled(modes)
    g = G.Grid((5, rows), lo=lo, hi=hi)
    g.set_state(st, t0=0.1, recon=True)
    before = g.read_state().astype(np.float64)
    g.step(G.Velocity("waves2d", modes=modes), dt, 1)
    after = g.read_state()
    g.close()
    ref = oracle.step(oracle.grid((5, rows), lo=lo, hi=hi), oracle.velocity("waves2d", modes=modes), before, 0.1, dt)
    assert np.max(np.abs(after[0] - ref[0])) <= 1e-5
    assert np.max(np.abs(after[1:3] - ref[1:3])) <= 1e-4


@pytest.mark.parametrize("layout", ["full", "compact"])
@pytest.mark.parametrize("n", [(5, 131071), (5, 600001), (1300, 1090)])
def test_run_equals_single_steps(G, n, layout):
    modes = inputs.wave_modes(64, seed=17)
    if n[0] == 5:
        h, lo, hi, st = _strip(n[1])
    else:
        h, lo, hi, st = 1.0 / (n[0] - 1), None, None, inputs.circle_sdf(n).astype(np.float32)
    dt = 0.8 * h / inputs.wave_speed_sampled(modes)
    vel = G.Velocity("waves2d", modes=modes)
    a, b = (G.Grid(n, lo=lo, hi=hi, layout=layout) for _ in range(2))
    for g in (a, b):
        g.set_state(st, t0=0.2, recon=True)
    a.step(vel, dt, 3)
    for _ in range(3):
        b.step(vel, dt, 1)
    ra, rb = a.read_state(), b.read_state()
    a.close()
    b.close()
    assert np.array_equal(ra, rb)
    assert np.isfinite(ra).all()
