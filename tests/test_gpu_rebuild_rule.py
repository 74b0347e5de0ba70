"""Which FULL 3D runs rebuild the mixed derivatives between their steps: not those of a constant
field whose every foot lies a whole cell away (the cells of a tile's last rows are then outside
it), nor a rotation's with the Euler trace on millions of nodes; either way a run equals single
steps bit for bit.  The rule shows in the launches: a step that rebuilds is one, a step that
reconstructs two, beside the run's coefficients and clock."""
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


SMALL, LARGE = (38, 41, 35), (130, 128, 128)
CASES = [
    # n, field, trace, cells per step (constant: along y), rebuilt
    (SMALL, "const", "rk3", 0.9, True), (SMALL, "const", "rk3", 1.0, False), (SMALL, "const", "euler", 1.0, False),
    (SMALL, "const", "rk3", 1.5, False), (SMALL, "rotation", "euler", 1.0, True), (SMALL, "rotation", "rk3", 1.0, True),
    (LARGE, "rotation", "euler", 1.0, False), (LARGE, "rotation", "rk3", 1.0, True), (LARGE, "const", "euler", 0.9, True),
    (LARGE, "deform3d", "euler", 1.0, True),
]


@pytest.mark.parametrize("n,kind,trace,cells,rebuilt", CASES)
def test_rule_and_bits(G, n, kind, trace, cells, rebuilt):
    st = inputs.sphere_sdf(n, center=(0.45, 0.5, 0.5), r=0.25).astype(np.float32)
    vel = G.Velocity(kind, trace=trace, omega=1.0, c=(0.6, -0.8, 0.5), T=3.0)
    # the constant field's y component; the fastest of the others over the unit box
    dt = cells / ((n[1] - 1) * 0.8) if kind == "const" else cells / (max(n) - 1) / dict(rotation=0.5, deform3d=2.0)[kind]
    a, b = G.Grid(n), G.Grid(n)
    for g in (a, b):
        g.set_state(st, t0=0.2, recon=True)
    steps = 5
    a.step(vel, dt, steps)
    assert a.last_step_launches() == 2 + (steps + 1 if rebuilt else 2 * steps)
    for _ in range(steps):
        b.step(vel, dt, 1)
    assert np.array_equal(a.read_state(), b.read_state())
    a.close()
    b.close()
