"""State planes to and from device arrays: one launch or copy calls, the same bits as through
host arrays for every alignment, row length, size and overlap of the arrays."""
import ctypes

import numpy as np
import pytest

from paper_0905_3409_gb300 import gals

pytestmark = pytest.mark.gpu


def _fields(shape, planes, seed=1):
    return np.random.default_rng(seed).standard_normal((planes,) + shape).astype(np.float32)


def _ptrs(addresses):
    return (ctypes.c_void_p * len(addresses))(*addresses)


# rows that are dense in the state (n0 a multiple of 4) and padded ones, one row of lanes and
# its remainder, planes of more than one pass of the largest launch (2^24 nodes)
SHAPES = [(4, 4), (7, 5), (64, 64), (33, 129), (509, 128), (33, 40000), (4100, 4100), (9, 6, 5), (32, 20, 12)]


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("shift", [0, 1, 4])
def test_device_arrays_match_host_arrays(n, shift):
    import torch

    g = gals.Grid(n)
    shape, P = tuple(reversed(n)), g.nplanes
    f = _fields(shape, P)
    g.set_state(f)
    size = int(np.prod(shape))
    stride = size + shift  # plane p starts at shift + p * stride floats of an aligned array
    out = torch.full((shift + P * stride,), 7.0, device="cuda")
    torch.cuda.synchronize()
    at = [out.data_ptr() + 4 * (shift + p * stride) for p in range(P)]
    gals._check(gals.lib().gals_read_state(g._h, _ptrs(at), P, gals.MEM_DEVICE), g._h)
    got = out.cpu().numpy()
    want = np.full_like(got, 7.0)
    for p in range(P):
        want[shift + p * stride: shift + p * stride + size] = f[p].ravel()
    np.testing.assert_array_equal(got, want)  # and nothing beside the planes
    h = gals.Grid(n)
    gals._check(gals.lib().gals_set_state(h._h, _ptrs(at), P, gals.MEM_DEVICE, ctypes.c_double(0.0), 0), h._h)
    np.testing.assert_array_equal(h.read_state(), f)


def test_arrays_that_overlap_and_page_locked_ones():
    import torch

    n = (96, 40)
    g = gals.Grid(n)
    f = _fields((40, 96), 4)
    g.set_state(f)
    out = torch.zeros((2, 40, 96), device="cuda")
    torch.cuda.synchronize()
    a, b = out[0].data_ptr(), out[1].data_ptr()
    # planes are written in order: the last one asked for stays
    gals._check(gals.lib().gals_read_state(g._h, _ptrs([a, a, b, a]), 4, gals.MEM_DEVICE), g._h)
    np.testing.assert_array_equal(out.cpu().numpy(), f[[3, 2]])
    pinned = torch.zeros((4, 40, 96)).pin_memory()
    gals._check(gals.lib().gals_read_state(g._h, _ptrs([pinned[p].data_ptr() for p in range(4)]), 4,
                                           gals.MEM_HOST), g._h)
    np.testing.assert_array_equal(pinned.numpy(), f)


def test_batch_reads_into_device_arrays():
    import torch

    sizes = [(64, 48), (33, 57), (128, 9)]
    b = gals.Batch(sizes)
    for k, s in enumerate(sizes):
        f = _fields((s[1], s[0]), 4, seed=k)
        src = torch.tensor(f, device="cuda")
        out = torch.zeros_like(src)
        torch.cuda.synchronize()
        gals._bcheck(gals.lib().gals_batch_set_state(b._h, k, _ptrs([src[p].data_ptr() for p in range(4)]), 4,
                                                     gals.MEM_DEVICE, ctypes.c_double(0.0), 0), b._h)
        gals._bcheck(gals.lib().gals_batch_read_state(b._h, k, _ptrs([out[p].data_ptr() for p in range(4)]), 4,
                                                      gals.MEM_DEVICE), b._h)
        np.testing.assert_array_equal(out.cpu().numpy(), f)
