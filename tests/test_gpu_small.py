"""Runs of 8 and more steps on a small 2D grid advance in one cluster launch with the state in
distributed shared memory; the result must equal one launch per step bit for bit: grids
of one to sixteen blocks, odd sides, rows that fill no pair, the size limit, feet that
cross several blocks, every velocity and trace, both layouts, approach B, mixed
derivatives given explicitly, odd and even step counts and a call longer than one run."""
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


def _vel(G, kind, trace="rk3"):
    kw = dict(vortex2d=dict(T=8.0), rotation=dict(omega=2 * math.pi), const=dict(c=(0.7, -0.4, 0.0)), pseudo1d={},
              fourier2d=dict(modes=inputs.fourier_modes(16, seed=31, periodic=True)) if kind == "fourier2d" else {},
              waves2d=dict(modes=inputs.wave_modes(24, seed=41)) if kind == "waves2d" else {})[kind]
    return G.Velocity(kind, trace=trace, **kw)


CASES = [
    # n, field, trace, cells per step at speed 1, layout, cross, steps, given phi_xy
    ((64, 64), "vortex2d", "rk3", 1.0, "full", "central", 9, False),
    ((64, 64), "vortex2d", "rk3", 1.0, "full", "central", 300, True),
    ((61, 47), "fourier2d", "rk3", 0.5, "compact", "central", 8, True),
    ((5, 4), "rotation", "rk3", 0.3, "full", "central", 8, False),
    ((24, 500), "fourier2d", "heun_psi", 0.5, "full", "central", 8, False),
    ((512, 24), "vortex2d", "euler", 1.0, "compact", "central", 11, False),
    ((111, 110), "rotation", "rk3", 4.0, "full", "cell", 9, False),      # feet 12 rows away
    ((130, 94), "const", "rk3", 2.0, "full", "central", 10, False),
    ((64, 33), "pseudo1d", "rk3", 0.5, "full", "cell", 9, False),
    ((80, 70), "waves2d", "heun_psi", 0.5, "compact", "central", 8, False),
]


@pytest.mark.parametrize("n,kind,trace,cells,layout,cross,steps,given", CASES)
def test_cluster_run_equals_single_steps(G, n, kind, trace, cells, layout, cross, steps, given):
    st = inputs.circle_sdf(n).astype(np.float32)
    if given:
        st[3] = np.random.default_rng(3).normal(size=st[3].shape)
    dt = cells / (max(n) - 1)
    vel = _vel(G, kind, trace)
    a, b = (G.Grid(n, layout=layout, cross=cross) for _ in range(2))
    for g in (a, b):
        g.set_state(st, t0=0.3, recon=not given)
    a.step(vel, dt, steps)
    # coefficients (and wave amplitudes), cluster kernel and clock of each run
    assert a.last_step_launches() == (4 if kind == "waves2d" else 3) * -(-steps // 256)
    for _ in range(steps):
        b.step(vel, dt, 1)
    assert np.array_equal(a.read_state(), b.read_state(), equal_nan=True)
    a.step(vel, dt, 8)
    for _ in range(8):
        b.step(vel, dt, 1)
    ra, rb = a.read_state(), b.read_state()
    assert np.array_equal(ra, rb, equal_nan=True)
    assert np.isfinite(ra[:3]).all()


def test_rule_edges(G):
    """One node row more than the limit, or a run of 7 steps, goes the general way; the results
    of the two ways agree bit for bit where a call's last run is short (256 + 7 steps)."""
    vel = _vel(G, "vortex2d")
    for n, steps, small in (((128, 96), 8, True), ((128, 97), 8, False), ((513, 20), 8, False), ((64, 64), 7, False)):
        a, b = G.Grid(n), G.Grid(n)
        for g in (a, b):
            g.set_state(inputs.circle_sdf(n).astype(np.float32), recon=True)
        a.step(vel, 0.5 / (max(n) - 1), steps)
        assert (a.last_step_launches() == 3) == small
        for _ in range(steps):
            b.step(vel, 0.5 / (max(n) - 1), 1)
        assert np.array_equal(a.read_state(), b.read_state())
    a, b = G.Grid((64, 64)), G.Grid((64, 64))
    for g in (a, b):
        g.set_state(inputs.circle_sdf((64, 64)).astype(np.float32), recon=True)
    a.step(vel, 1.0 / 63, 263)
    for _ in range(263):
        b.step(vel, 1.0 / 63, 1)
    assert np.array_equal(a.read_state(), b.read_state())
