"""Device-array reads and writes of a state with few, long rows (a wide 2D strip, a wide slab):
the same bits as through host arrays at the edges of the pieces that a row is split into, and
no slower than rows of ordinary length by more than a small factor (a row per warp made a
read of 10^6 x 4 nodes 39 times slower than copy calls)."""
import time

import numpy as np
import pytest

from paper_0905_3409_gb300 import gals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(511, 4), (513, 5), (1023, 4), (1537, 7), (1000001, 4), (100003, 16), (50001, 5, 5)])
def test_long_rows_match_host_arrays(n):
    import torch

    shape, P = tuple(reversed(n)), 2 ** len(n)
    f = np.random.default_rng(3).standard_normal((P,) + shape).astype(np.float32)
    a, b = gals.Grid(n), gals.Grid(n)
    a.set_state(torch.tensor(f, device="cuda"))
    b.set_state(f)
    out = torch.full((P + 1,) + shape, 7.0, device="cuda")  # and nothing behind the planes
    a.read_state(out, nfields=P)
    np.testing.assert_array_equal(out[:P].cpu().numpy(), f)
    assert bool((out[P] == 7.0).all())
    np.testing.assert_array_equal(a.read_state(), b.read_state())
    for g in (a, b):
        g.close()


def test_long_rows_are_copied_by_many_warps():
    import torch

    def best(n):
        g = gals.Grid(n)
        out = torch.zeros((3,) + tuple(reversed(n)), device="cuda")
        g.set_state(out)
        t = []
        for _ in range(10):
            t0 = time.perf_counter()
            g.read_state(out, nfields=3)
            t.append(time.perf_counter() - t0)
        g.close()
        return min(t)

    assert best((1000001, 4)) <= 5 * best((2001, 2000))
