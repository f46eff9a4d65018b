"""What lbm_config_describe says of the generic kernel (configuration 0): the
threads of a CTA as it is launched.  Host code: no GPU."""
import ctypes

import pytest


def threads(lbm, nx, ny, precision):
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", precision)
    t, s, n = ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
    assert lbm.lbm_config_describe(ctypes.byref(p), 0, ctypes.byref(t), ctypes.byref(s), ctypes.byref(n)) == 0
    assert (s.value, n.value) == (0, 1)
    return t.value


@pytest.mark.parametrize("nx,ny", [(1023, 1021), (4096, 4096), (1, 131072)])
def test_fp32_walks_of_tiles(lbm, nx, ny):
    """Eight warps of a 32 x 8 tile and two of its ring, from 2^17 nodes."""
    assert threads(lbm, nx, ny, "fp32") == 320


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tiles(lbm, precision):
    """A warp for the one node and one for its ring; whole warps, at most 384 threads, elsewhere."""
    assert threads(lbm, 1, 1, precision) == 64
    for nx, ny in ((64, 64), (256, 256), (3, 400), (301, 17)):
        t = threads(lbm, nx, ny, precision)
        assert t % 32 == 0 and 64 <= t <= 384
