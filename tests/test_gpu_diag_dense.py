"""Diagnostics of states most of whose cells the bound cannot decide (noise, large slopes): a warp's
few undecided cells are sampled where they are found, many of them from a list, and past the
list by sampling the whole grid.  The counts must be the same whichever way a cell goes:
those of a grid against the sum over strips of it, exactly, in 2D and 3D, for both ways of the
mixed derivatives, sample counts below and above a warp, narrow and wide grids, and bands of noise of every extent in a smooth
state; thinned noise (few undecided cells a warp) against the same cells in noise; and
against FP64 sampling.  The time of such a state is bounded by that of a smooth
one (a warp per cell made them thirteen times slower, and slower than sampling every cell)."""
import itertools
import time

import numpy as np
import pytest

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


def _noise(n, seed, band=None):
    """O(1) noise in every plane (spacing 1); band: rows outside [a, b) hold phi = 1 alone."""
    st = np.random.default_rng(seed).normal(size=(2 ** len(n),) + tuple(reversed(n))).astype(np.float32)
    if band:
        for sl in (slice(0, band[0]), slice(band[1], None)):
            st[:, sl] = 0.0
            st[0, sl] = 1.0
    return st


def _counts(G, a, b, q, cross):
    """(n_negative, n_symdiff, n_negative without a reference) on a grid of spacing 1."""
    n = a.shape[:0:-1]
    ga, gb = (G.Grid(n, lo=(0.0,) * len(n), hi=tuple(m - 1.0 for m in n), cross=cross) for _ in range(2))
    ga.set_state(a)
    gb.set_state(b)
    d, alone = ga.diagnostics(q=q, reference=gb), ga.diagnostics(q=q)
    ga.close()
    gb.close()
    assert alone["n_symdiff"] == 0
    return np.array([d["n_negative"], d["n_symdiff"], alone["n_negative"]], dtype=np.int64)


@pytest.mark.parametrize("n,q,band,cross,strip", [
    ((701, 303), 1, None, "central", 8), ((701, 303), 2, None, "cell", 8), ((701, 303), 4, None, "central", 8),
    ((701, 303), 7, None, "cell", 8),
    # of 6688 warps an eighth, 836, may be in the list: bands of 25, 36 and 41 rows of 22
    ((701, 303), 4, (100, 125), "central", 8), ((701, 303), 4, (100, 136), "cell", 8),
    ((701, 303), 2, (100, 141), "central", 8),
    ((5, 9000), 3, None, "central", 100), ((9, 4000), 1, None, "cell", 100), ((17, 3000), 2, None, "central", 100),
    ((33, 2000), 4, None, "central", 60), ((4, 4), 2, None, "central", 4),
    ((40, 36, 60), 1, None, "central", 4), ((40, 36, 60), 2, None, "cell", 4), ((40, 36, 60), 3, None, "central", 4),
    ((70, 5, 200), 5, None, "cell", 20),
])
def test_counts_do_not_depend_on_the_way(G, n, q, band, cross, strip):
    a, b = _noise(n, 1, band), _noise(n, 2, band)
    whole = _counts(G, a, b, q, cross)
    parts = np.zeros(3, np.int64)
    for r in range(0, n[-1] - 1, strip):             # strips share a row of nodes and no cell
        parts += _counts(G, *(np.ascontiguousarray(s[:, r:r + strip + 1]) for s in (a, b)), q, cross)
    assert np.array_equal(whole, parts), (whole, parts)


@pytest.mark.parametrize("q", [1, 2, 3, 4, 7])
@pytest.mark.parametrize("n", [(701, 303), (70, 36, 40)])
def test_few_undecided_cells_a_warp(G, n, q):
    """Columns of noise 16 apart, two cells wide, in phi = 1 (a few undecided cells a warp), against
    the strips of four columns around them, whose narrow grids make every warp dense."""
    a, b = _noise(n, 1), _noise(n, 2)
    cols = np.arange(n[0]) % 16 == 7
    for st in (a, b):
        st[:, ..., ~cols] = 0.0
        st[0, ..., ~cols] = 1.0
    whole = _counts(G, a, b, q, "central")
    parts = np.zeros(3, np.int64)
    for c in np.flatnonzero(cols):
        parts += _counts(G, *(np.ascontiguousarray(s[..., c - 2:c + 2]) for s in (a, b)), q, "central")
    assert np.array_equal(whole, parts), (whole, parts)


def _weights(xi):
    o = 1 - xi
    return [(o * o * (1 + 2 * xi), xi * o * o), (xi * xi * (3 - 2 * xi), -xi * xi * o)]


@pytest.mark.parametrize("n,q", [((701, 303), 2), ((40, 36, 60), 2)])
def test_counts_against_fp64(G, n, q):
    dim = len(n)
    plane = {2: [(0, 0), (1, 0), (0, 1), (1, 1)],
             3: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1)]}[dim]
    H = []
    a, b = _noise(n, 1), _noise(n, 2)
    for st in (a, b):
        out = []
        for s in itertools.product(range(q), repeat=dim):
            W = [_weights((k + 0.5) / q) for k in s]
            h = 0.0
            for c in itertools.product((0, 1), repeat=dim):
                sl = tuple(slice(e, e + m - 1) for e, m in zip(reversed(c), reversed(n)))
                for p, o in enumerate(plane):
                    h = h + np.prod([W[d][c[d]][o[d]] for d in range(dim)]) * st[p][sl].astype(np.float64)
            out.append(h)
        H.append(np.stack(out))
    near = [np.abs(h) <= 60 * 6e-8 * 4 * np.abs(st).max() for h, st in zip(H, (a, b))]  # FP32 rounding
    neg, sym, _ = _counts(G, a, b, q, "central")
    assert abs(neg - int((H[0] < 0).sum())) <= int(near[0].sum())
    assert abs(sym - int(((H[0] < 0) != (H[1] < 0)).sum())) <= int((near[0] | near[1]).sum())


@pytest.mark.parametrize("q", [1, 2, 4])
def test_noise_costs_a_small_factor(G, q):
    import torch

    n = (2048, 2048)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    noise = torch.randn((4,) + n, device="cuda", generator=gen)
    smooth = torch.zeros((4,) + n, device="cuda")
    smooth[0] = torch.linspace(-1.0, 2.0, n[0], device="cuda")

    def best(st):
        a, b = (G.Grid(n, lo=(0.0, 0.0), hi=(2047.0, 2047.0)) for _ in range(2))
        a.set_state(st)
        b.set_state(st.flip(-1).contiguous())
        t = []
        for _ in range(8):
            t0 = time.perf_counter()
            a.diagnostics(q=q, reference=b)
            t.append(time.perf_counter() - t0)
        a.close()
        b.close()
        return min(t)

    assert best(noise) <= 6 * best(smooth)
