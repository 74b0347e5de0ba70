"""The fused training step (batches of at most 16384 samples: forward and backward pass of a
chunk per block) at the edges of its chunks: one sample, chunks of 128 and fewer rows, a
ragged last chunk, the largest fused batch and the smallest general one.  Gradients against
the FP64 oracle network within 4e-2 per tensor (the deepest path has ten products of two
BF16 operands, each rounded by at most 2^-9: 20 x 2^-9 = 3.9e-2), and the two paths against each other: the gradient of a batch and of the same
batch repeated to a size that the general path takes differ by rounding only."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SIZES = [3, 128, 128, 128, 128, 6]


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    from paper_0905_3409_gb300 import gals
    return gals


def _data(n, seed=0):
    rng = np.random.default_rng(seed)
    return rng.uniform(-1, 1, (n, 3)).astype(np.float32), rng.normal(size=(n, 6)).astype(np.float32)


def _tensors(g):
    at = 0
    for i, o in zip(SIZES[:-1], SIZES[1:]):
        yield g[at:at + i * o]
        yield g[at + i * o:at + i * o + o]
        at += i * o + o


@pytest.mark.parametrize("n", [1, 127, 128, 129, 1013, 16384])
def test_fused_gradient_matches_oracle(G, n):
    S = G.Surrogate(seed=5)
    p, _ = S.get_params()
    X, T = _data(n, seed=n)
    loss, grad = S.gradient(X, T)
    rloss, rgrad = oracle.mlp_backward(SIZES, p.astype(np.float64), X.astype(np.float64), T.astype(np.float64))
    assert loss == pytest.approx(rloss, rel=4e-2)
    for a, b in zip(_tensors(grad), _tensors(rgrad)):
        assert np.linalg.norm(a - b) <= 4e-2 * np.linalg.norm(b)


def test_fused_and_general_paths_agree(G):
    """4 x 5000 repeated samples go the general way, 5000 the fused one.  Every product is of
    the same BF16 operands; only the FP32 sums over samples run in another order (at most
    20000 terms: 1e-5 of the gradient's norm is 4 standard deviations of such a sum's
    rounding for tensors whose terms do not cancel below a hundredth)."""
    S = G.Surrogate(seed=5)
    X, T = _data(5000, seed=7)
    l1, g1 = S.gradient(X, T)
    l2, g2 = S.gradient(np.tile(X, (4, 1)), np.tile(T, (4, 1)))
    assert abs(l1 - l2) <= 1e-12 * abs(l1)
    for a, b in zip(_tensors(g1), _tensors(g2)):
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)


def test_sample_groups_do_not_change_the_training(G):
    """A launch makes the samples of several steps: training 20 steps of a batch whose groups
    hold 16 steps equals the same steps taken by two surrogates from the same weights (10
    steps, whose one group is shorter)."""
    from paper_0905_3409_gb300 import inputs
    modes = inputs.fourier_modes(16, periodic=True)
    vel = G.Velocity("fourier2d", modes=modes)
    h = 1.0 / 255
    dt = h / inputs.fourier_speed_bound(modes)
    out = []
    for steps in (20, 20, 3):
        S = G.Surrogate(seed=9)
        r = S.train(vel, dt, h, steps=steps, batch=16384, lr=1e-3, lr_min=1e-3)
        out.append((S.get_params()[0], r))
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1]["initial_loss"] == pytest.approx(out[2][1]["initial_loss"], rel=1e-12)
