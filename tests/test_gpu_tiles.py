"""The generic step's tiles at the sizes where their cut can go wrong: one
node, single rows and columns (the ring wraps onto the tile itself), prime
sides (tiles of unequal size), and lattices of many tiles.

FP64 against the oracle at the parity bar (1e-12 of the largest population);
FP32 at the element-wise bar of 2e-5 on the density.
"""
import numpy as np
import pytest

import oracle
from paper_1412_5170_gb300 import synth

pytestmark = pytest.mark.gpu
MRT = dict(s_e=0.8, s_eps=0.8, s_q=1.1)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("coll,forc", [("mrt", "guo"), ("bgk", "edm")])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 331), (331, 1), (2, 97), (67, 3), (31, 257), (263, 129)])
def test_tiles(lbm, nx, ny, coll, forc, precision):
    rv, rl = lbm.maxwell(0.8)
    rho0 = synth.density_field(nx, ny, "droplet", rl, rv, max(1.5, min(nx, ny) / 4), seed=5)
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, coll, forc, precision, **MRT)
    with lbm.Lattice(p) as lat:
        lat.variant = 0
        lat.init_density(rho0)
        lat.step(25)
        f, st = lat.read_populations(), lat.stats()
    ref, ost = oracle.run(oracle.params(nx, ny, 0.8, 0.9, -0.304, 1.0, coll, forc, **MRT), oracle.init_rest(rho0), 25)
    assert ost == 0 and st["status"] == 0
    if precision == "fp64":
        assert np.abs(f - ref).max() < 1e-12 * np.abs(ref).max()
    else:
        assert (np.abs(f.sum(0) - ref.sum(0)) / ref.sum(0)).max() < 2e-5


# 2^17 nodes and more: walks of 32 x 8 tiles; ragged last strips and chunks,
# strips of one column (1057 = 33 * 32 + 1), fewer columns than a strip
@pytest.mark.parametrize("coll,forc", [("mrt", "guo"), ("bgk", "guo"), ("bgk", "edm"), ("bgk", "sc"), ("bgk", "li")])
@pytest.mark.parametrize("nx,ny", [(379, 361), (1057, 129), (31, 4231), (4231, 33)])
def test_tile_walks(lbm, nx, ny, coll, forc):
    rv, rl = lbm.maxwell(0.8)
    rho0 = synth.density_field(nx, ny, "droplet", rl, rv, min(nx, ny) / 4, seed=5)
    A, sigma = (0.0, 0.105) if forc == "li" else (-0.304, 0.0)
    p = lbm.make_params(nx, ny, 0.8, 0.9, A, 1.0, coll, forc, "fp32", sigma=sigma, **MRT)
    with lbm.Lattice(p) as lat:
        assert lat.config == 0
        lat.init_density(rho0)
        lat.step(10)
        f, st = lat.read_populations(), lat.stats()
    ref, ost = oracle.run(oracle.params(nx, ny, 0.8, 0.9, A, 1.0, coll, forc, sigma=sigma, **MRT), oracle.init_rest(rho0), 10)
    assert ost == 0 and st["status"] == 0
    assert (np.abs(f.sum(0) - ref.sum(0)) / ref.sum(0)).max() < 2e-5
    assert np.abs(f - ref).max() < 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("precision,nx,ny", [("fp64", 1024, 1024), ("fp32", 512, 4096), ("fp32", 1536, 1536)])
def test_injected_timeout_where_the_generic_kernel_is_the_automatic_choice(lbm, precision, nx, ny):
    """Generic kernel by default, but strips fill the GPU too, so the step of
    the injection takes them; a caller's choice of the generic kernel, and a
    lattice that strips do not fill, refuse it."""
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "mrt", "guo", precision, **MRT)
    with lbm.Lattice(p) as lat:
        assert lat.config == 0
        lat.init_preset("droplet", 100.0)
        lat.step(2)
        lat.inject_stage_timeout()
        lat.step(1)
        assert lat.stats()["status"] == lbm.E_TIMEOUT
        lat.init_preset("droplet", 100.0)
        lat.step(3)
        assert lat.stats()["status"] == 0
        lat.variant = 0
        with pytest.raises(lbm.LbmError):
            lat.inject_stage_timeout()
    with lbm.Lattice(lbm.make_params(64, 64, 0.8, 0.9, -0.304, 1.0, "mrt", "guo", precision, **MRT)) as lat:
        with pytest.raises(lbm.LbmError):
            lat.inject_stage_timeout()
