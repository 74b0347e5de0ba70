"""2D steps that write no phi_xy plane (between the steps of a run, COMPACT, approach B) on the
two tile shapes: short tiles on grids with fewer than about a wave of tall ones, tall
walked tiles above.  Whatever the shape, a run of steps must equal single steps (which
write phi_xy and use the exchanging tiles in the FULL layout) bit for bit, and a step of
the tall tiles must equal the short tiles' on the same rows."""
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


def _vel(G, kind, trace):
    modes = inputs.fourier_modes(16, seed=31, periodic=True) if kind == "fourier2d" else (
        inputs.wave_modes(8, seed=41) if kind == "waves2d" else None)
    return G.Velocity(kind, trace=trace, T=8.0, omega=2 * math.pi, c=(0.6, -0.8, 0.0), modes=modes)


# n on both sides of the tile rule (850 tiles of 128 x 14): 1300 x 1060 is 836 tiles, 1300 x 1090
# 858; a last tile of one column (1281) and a last row alone (1093 = 78 * 14 + 1)
@pytest.mark.parametrize("n,kind,trace,cfl,layout,cross", [
    ((1300, 1060), "vortex2d", "rk3", 1.0, "full", "central"),
    ((1300, 1090), "vortex2d", "rk3", 1.0, "full", "central"),
    ((1281, 1093), "rotation", "rk3", 2.5, "full", "central"),
    ((1281, 1093), "vortex2d", "heun_psi", 1.0, "compact", "central"),
    ((1282, 1091), "vortex2d", "rk3", 1.0, "full", "cell"),
    ((1285, 1107), "const", "euler", 3.0, "full", "central"),
    ((1310, 1100), "fourier2d", "rk3", 0.5, "full", "central"),
    ((1300, 1090), "waves2d", "rk3", 0.5, "compact", "central"),
    ((301, 5), "rotation", "rk3", 0.5, "full", "central"),
])
def test_run_equals_single_steps_on_both_tile_shapes(G, n, kind, trace, cfl, layout, cross):
    st = inputs.circle_sdf(n).astype(np.float32)
    vel = _vel(G, kind, trace)
    dt = cfl / (max(n) - 1) / (math.pi if kind == "rotation" else 1.0)
    a, b = (G.Grid(n, layout=layout, cross=cross) for _ in range(2))
    for g in (a, b):
        g.set_state(st, t0=0.2, recon=True)
    a.step(vel, dt, 5)
    for _ in range(5):
        b.step(vel, dt, 1)
    ra, rb = a.read_state(), b.read_state()
    assert np.array_equal(ra, rb, equal_nan=True)
    assert np.isfinite(ra).all()


def test_tall_tiles_equal_short_tiles(G):
    """The same columns on a grid whose tiles are short and as part of a taller grid of the
    same spacing whose tiles are tall (constant velocity: no position enters the trace)."""
    nx, small, large = 257, 900, 4200      # 195 and 900 tiles of 128 x 14
    st = inputs.random_state((4, large, nx), seed=5).astype(np.float32)
    vel = _vel(G, "const", "rk3")
    out = []
    for ny in (small, large):
        g = G.Grid((nx, ny), lo=(0.0, 0.0), hi=(256.0, float(ny - 1)), layout="compact")
        g.set_state(np.ascontiguousarray(st[:, :ny]), recon=True)
        g.step(vel, 0.7, 3)
        out.append(g.read_state()[:3, : small - 10])
        g.close()
    assert np.array_equal(out[0], out[1])
