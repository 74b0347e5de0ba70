"""The residual check of the learned trace runs beside the network, one tile behind: every
tile ends as the network's or the exact trace's, whole, and the counters say how many."""
import numpy as np
import pytest

from paper_0905_3409_gb300 import gals, inputs

pytestmark = pytest.mark.gpu


# one tile; fewer tiles than groups; ragged rows; more tiles than one round of the chip
@pytest.mark.parametrize("n", [(5, 4), (129, 4), (300, 200), (1100, 260)])
@pytest.mark.parametrize("field", ["fourier2d", "waves2d"])
@pytest.mark.parametrize("samples", [1, 4, 33, 128])
def test_tiles_are_learned_or_exact(n, field, samples):
    modes = inputs.fourier_modes(16, seed=5, periodic=True) if field == "fourier2d" else inputs.wave_modes(24, seed=5)
    h = 1.0 / 256
    speed = inputs.fourier_speed_bound(modes) if field == "fourier2d" else inputs.wave_speed_sampled(modes)
    dt = h / speed
    vel = gals.Velocity(field, modes=modes)
    S = gals.Surrogate(seed=2)
    S.bind(vel, dt, h)  # random weights: a wrong map, by an amount that varies over the box
    learned = gals.Velocity(field, modes=modes, trace="surrogate", surrogate=S)
    x, y = np.meshgrid(h * np.arange(n[0]), h * np.arange(n[1]))
    r = np.hypot(x + 0.2, y + 0.1)
    state = np.stack([r - 0.5, (x + 0.2) / r, (y + 0.1) / r]).astype(np.float32)
    g = gals.Grid(n, hi=[h * (n[0] - 1), h * (n[1] - 1)])
    tiles = (n[0] + 127) // 128 * n[1]

    def step(v, tol):
        S.set_check(tol_x=tol, tol_J=1e9 if tol else 0.0, samples=samples)
        S.stats(reset=True)
        g.set_state(state, t0=0.3)
        g.step(v, dt, 1)
        return g.read_state(nfields=3), S.stats()

    net, (t, f) = step(learned, 1e9)
    assert (t, f) == (tiles, 0)
    exact, (t, f) = step(learned, 0.0)
    assert (t, f) == (tiles, tiles)
    # the exact trace of the step kernel itself: two FP32 evaluations of the same RK3 trace, at
    # CFL 1 a few rounding errors of phi (|grad phi| = 1, values below 5) and of H'/h apart
    plain, _ = step(vel, 1.0)
    assert np.max(np.abs(exact[0] - plain[0])) <= 8 * 2.0 ** -22
    assert np.max(np.abs(exact[1:] - plain[1:])) <= 1.5 * 256 * 8 * 2.0 ** -22
    for tol in (0.1, 0.3, 0.6, 0.9):
        mixed, (t, f) = step(learned, tol)
        assert t == tiles
        failed = 0
        for b in range(0, n[0], 128):
            part = np.s_[:, :, b:b + 128]
            is_net = (mixed[part] == net[part]).all(axis=(0, 2))
            is_exact = (mixed[part] == exact[part]).all(axis=(0, 2))
            assert (is_net | is_exact).all()
            assert not (is_net & is_exact).any()
            failed += int(is_exact.sum())
        assert failed == f
