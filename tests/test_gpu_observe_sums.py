"""Sums of the observables from walks of tiles: FP64 for FP32 deviations too,
so an infinite density gives an infinite mass (a float pair's error term made
it NaN), whatever the width."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(33, 9), (36, 9), (1, 64), (381, 361)])
def test_infinite_density(lbm, nx, ny, precision):
    rv, rl = lbm.maxwell(0.8)
    rho0 = np.full((ny, nx), rv)
    rho0[ny // 3, nx // 3] = np.inf
    with lbm.Lattice(lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", precision)) as lat:
        lat.init_density(rho0)
        st = lat.stats()
    assert st["status"] == lbm.E_NONFINITE and st["mass"] == np.inf and st["rho_max"] == np.inf
