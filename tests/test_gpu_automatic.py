"""The automatic kernel choice of FP32 lattices, and what it steps with at the
shapes where the choice changes: strips of 1024 and of 512 columns that do not
divide the width, the generic walk where neither covers it, flat lattices.

Every choice evaluates the same update per node: 2e-5 of the density after
ten steps against the generic kernel (the FP32 element-wise bar)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MRT = dict(s_e=0.8, s_eps=0.8, s_q=1.1)


def params(lbm, nx, ny, coll="mrt"):
    return lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, coll, "guo", "fp32", **MRT)


def shape(lat):
    """Columns of the automatic choice's strips and their stages; 0 for the generic kernel."""
    cfg = lat.config
    assert cfg in (0, 8, 11, 12)   # the generic kernel and the carried block strips
    return (0, 0) if cfg == 0 else (4 * lat.configs()[cfg][1], lat.configs()[cfg][2])


# a strip of 1024 columns up to a fifth idle, 512 where these cover better, the walk elsewhere and below 2^22 nodes
@pytest.mark.parametrize("nx,ny,want", [(4096, 4096, (1024, 2)), (3840, 4096, (1024, 2)), (3712, 4096, (1024, 2)), (2888, 4096, (1024, 2)),
                                        (1924, 4096, (1024, 2)), (900, 8192, (1024, 2)), (1536, 4096, (512, 2)), (2432, 4096, (512, 2)),
                                        (512, 8192, (512, 3)), (512, 16384, (512, 2)), (2176, 4096, (0, 0)), (1100, 4096, (0, 0)),
                                        (64, 65536, (0, 0)), (2047, 4096, (0, 0)), (2044, 2048, (0, 0)), (400000, 3, (1024, 2)),
                                        (200000, 7, (1024, 2)), (100000, 7, (0, 0)), (400001, 3, (0, 0))])
def test_choice(lbm, nx, ny, want):
    with lbm.Lattice(params(lbm, nx, ny)) as lat:
        assert shape(lat) == want, (nx, ny)


@pytest.mark.parametrize("nx,ny", [(3588, 1180), (1928, 2200), (900, 4700), (1532, 2750), (508, 8300), (2176, 1930), (200000, 3)])
def test_choice_steps_like_the_generic_kernel(lbm, nx, ny):
    rv, rl = lbm.maxwell(0.8)
    out = []
    for variant in (-1, 0):
        with lbm.Lattice(params(lbm, nx, ny)) as lat:
            lat.variant = variant
            lat.init_preset("droplet_array", min(nx, ny) / 8, cell=max(8, min(nx, ny) // 3), seed=3)
            lat.step(10)
            st = lat.stats()
            assert st["status"] == 0
            out.append(lat.read_moments()[0])
    assert (np.abs(out[0] - out[1]) / out[1]).max() < 2e-5
