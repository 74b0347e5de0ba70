"""The diagnostics decide most cells by a bound on their corner data and sample only the rest.
The counts must be those of sampling every cell: on states whose interface passes through
cells in every way (noise at the scale of a cell, gradients that turn the sign between
corners of one sign, values exactly 0), with NaN and infinities in any plane, in 2D and 3D,
for both ways of the mixed derivatives and sample counts that do not fill a warp; the
reference counts are numpy's in FP64, and a sample whose value is within FP32 rounding of 0
may fall either way."""
import itertools

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


def _weights(xi, h):
    o = 1 - xi
    return [(o * o * (1 + 2 * xi), h * xi * o * o), (xi * xi * (3 - 2 * xi), -h * xi * xi * o)]


PLANES = {2: {(0, 0): 0, (1, 0): 1, (0, 1): 2, (1, 1): 3},
          3: {(0, 0, 0): 0, (1, 0, 0): 1, (0, 1, 0): 2, (0, 0, 1): 3, (1, 1, 0): 4, (1, 0, 1): 5, (0, 1, 1): 6,
              (1, 1, 1): 7}}


def _samples(st, q):
    """H at every sample of every cell (q^dim, cells...) in FP64."""
    dim = st.ndim - 1
    n = st.shape[:0:-1]
    h = [1.0 / (m - 1) for m in n]
    out = []
    for s in itertools.product(range(q), repeat=dim):
        W = [_weights((k + 0.5) / q, hh) for k, hh in zip(s, h)]
        H = 0.0
        for c in itertools.product((0, 1), repeat=dim):
            sl = tuple(slice(e, e + m - 1) for e, m in zip(reversed(c), reversed(n)))
            for a in itertools.product((0, 1), repeat=dim):
                w = np.prod([W[d][c[d]][a[d]] for d in range(dim)])
                H = H + w * st[PLANES[dim][a]][sl].astype(np.float64)
        out.append(H)
    return np.stack(out)


def _state(n, seed, kind):
    rng = np.random.default_rng(seed)
    dim = len(n)
    h = 1.0 / (max(n) - 1)
    shape = (2 ** dim,) + tuple(reversed(n))
    st = rng.normal(size=shape).astype(np.float32)
    order = {0: 0, 1: 1, 2: 1, 3: 1 if dim == 3 else 2, 4: 2, 5: 2, 6: 2, 7: 3}
    for p in range(2 ** dim):
        st[p] /= np.float32(h ** order[p])          # slopes that matter within a cell
    if kind == "shifted":                            # mostly one sign, turned by the slopes in places
        st[0] = np.abs(st[0]) + np.float32(0.6)
    if kind == "zeros":
        st[:, :: 2] = 0.0
    if kind == "smooth":
        x = np.linspace(0, 1, n[0])
        st[:] = 0
        st[0] = (x - 0.4).astype(np.float32)
        st[1] = 1.0
    return st


@pytest.mark.parametrize("n,q,kind", [((65, 33), 4, "noise"), ((100, 7), 3, "shifted"), ((31, 130), 16, "shifted"),
                                      ((64, 64), 2, "zeros"), ((257, 130), 5, "smooth"), ((4, 4), 1, "noise"),
                                      ((17, 9, 12), 3, "noise"), ((33, 8, 7), 2, "shifted"), ((9, 10, 11), 5, "smooth")])
def test_counts_match_sampling_every_cell(G, n, q, kind):
    a, b = _state(n, 1, kind), _state(n, 2, kind)
    ga, gb = G.Grid(n), G.Grid(n)
    ga.set_state(a)
    gb.set_state(b)
    d = ga.diagnostics(q=q, reference=gb)
    Ha, Hb = _samples(a, q), _samples(b, q)
    # FP32: at most about 60 roundings of terms of the sample's magnitude
    near = [np.abs(H) <= 60 * 6e-8 * np.abs(s).max() * 4 for H, s in ((Ha, a[0]), (Hb, b[0]))]
    if kind == "zeros":
        near = [np.zeros_like(m) for m in near]      # exact zeros are exact in FP32 too
        near = [m | ((H != 0) & (np.abs(H) <= 1e-5)) for m, H in zip(near, (Ha, Hb))]
    assert abs(d["n_negative"] - int((Ha < 0).sum())) <= int(near[0].sum())
    assert abs(d["n_symdiff"] - int(((Ha < 0) != (Hb < 0)).sum())) <= int((near[0] | near[1]).sum())
    alone = ga.diagnostics(q=q)
    assert alone["n_negative"] == d["n_negative"] and alone["n_symdiff"] == 0


@pytest.mark.parametrize("dim", [2, 3])
def test_not_finite_values_are_sampled(G, dim):
    """A NaN or an infinity in any plane of a corner: the cell's samples count as the FP32
    evaluation says (NaN < 0 is false), whatever the other corners are."""
    n = (12, 11) if dim == 2 else (12, 11, 10)
    for p in range(2 ** dim):
        for v in (np.nan, np.inf, -np.inf):
            st = np.zeros((2 ** dim,) + tuple(reversed(n)), np.float32)
            st[0] = -1.0
            st[(p,) + (5,) * dim] = v
            g = G.Grid(n)
            g.set_state(st)
            d = g.diagnostics(q=2)
            cells = int(np.prod([m - 1 for m in n]))
            touched = 2 ** dim * 2 ** dim  # samples of the cells around the node
            assert d["nonfinite"] == 1
            assert cells * 2 ** dim - touched <= d["n_negative"] <= cells * 2 ** dim
            if np.isnan(v):
                assert d["n_negative"] == cells * 2 ** dim - touched
            g.close()
