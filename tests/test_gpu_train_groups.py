"""Training draws the samples of several steps per launch (16 steps of 16384 samples).  Whatever
the group, step k trains on the samples of step k: the loss that a training of k steps
reports last is the loss of step k's samples with the weights after k - 1 steps, for steps
inside the first group, at its end, at the start of the next ones and in a short last group.
The samples are made here (the SplitMix64 stream of (seed, step, sample)), their targets by
gals_surrogate_targets (the training's own FP32 flow map), the loss by
gals_surrogate_gradient (the training's own products).  Weights: a training of k - 1 steps
takes the same first k - 1 steps, in groups of another length (one group of k - 1 against
16 and a rest, the learning rate constant).

Tolerance: the inputs are the same bits; a target's difference from the training's is that
of two compilations of one FP32 flow map (an ulp of J, 6e-8 / dt = 6e-5 of targets of O(10),
of either sign) and the rounding of the divisions (a few 2^-24), so that a mean over 98304
squares moves by about 1e-5 / sqrt(98304) of itself at random and a few 1e-7 in one
direction: 1e-5 of the loss leaves a factor of ten.  Another step's
samples move the loss by its sampling error, about 1/sqrt(6 x 16384) of it, now and then by
chance less: a second test asks that any one wrong order is ten tolerances away at one of
the steps."""
import numpy as np
import pytest

from paper_0905_3409_gb300 import inputs

pytestmark = pytest.mark.gpu

SEED, N = 771, 16384
STEPS = [1, 2, 16, 17, 18, 32, 33, 37]


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    from paper_0905_3409_gb300 import gals
    return gals


def _uniform(key):
    """The top 24 bits of SplitMix64's output for each 64-bit key, as a fraction."""
    with np.errstate(over="ignore"):
        z = key + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(40)).astype(np.float32) * np.float32(2.0 ** -24)


def _points(step):
    with np.errstate(over="ignore"):
        key = np.uint64(SEED) * np.uint64(0x100000001B3) ^ np.uint64(step << 24) ^ np.arange(N, dtype=np.uint64) * np.uint64(4)
    return np.stack([_uniform(key + np.uint64(c)) for c in range(3)], axis=1)


@pytest.fixture(scope="module")
def losses(G):
    """Per k: the loss that a training of k steps reports last, and a function of the loss on
    the samples of any step with the weights of that step's start."""
    modes = inputs.fourier_modes(16, periodic=True)
    vel = G.Velocity("fourier2d", modes=modes)
    h = 1.0 / 255
    dt = h / inputs.fourier_speed_bound(modes)
    opts = dict(batch=N, lr=1e-3, lr_min=1e-3, seed=SEED)

    def of(k):
        S = G.Surrogate(seed=9)
        reported = S.train(vel, dt, h, steps=k, **opts)["final_loss"]
        scales = S.get_params()[1]
        before = G.Surrogate(seed=9)
        if k > 1:
            before.train(vel, dt, h, steps=k - 1, **opts)

        def loss(step):
            P = _points(step)
            T = before.targets(vel, dt, h, P) / scales
            return before.gradient(2 * P - np.float32(1), T)[0]

        return reported, loss

    return {k: of(k) for k in STEPS}


@pytest.mark.parametrize("k", STEPS)
def test_step_k_trains_on_the_samples_of_step_k(losses, k):
    reported, loss = losses[k]
    own = loss(k)
    assert abs(reported - own) <= 1e-5 * own, (reported, own)


@pytest.mark.parametrize("other", [lambda k: 1, lambda k: k - 1, lambda k: k + 1, lambda k: k - 16,
                                   lambda k: (k - 1) % 16 + 1])
def test_other_samples_would_show(losses, other):
    """Of every wrong order of the samples, at one of the steps at least."""
    apart = [abs(loss(other(k)) / loss(k) - 1) for k, (_, loss) in losses.items() if 1 <= other(k) != k]
    assert max(apart) >= 1e-4
