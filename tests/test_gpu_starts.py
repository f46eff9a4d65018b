"""A start at rest and the built-in fields on shapes where the node walk of
their kernels carries from row to row in different ways: rows much shorter
than the grid, rows longer than it, one column, one row.

rho0 comes back from the moments: the nine products w_a rho0 and their sum
round eighteen times (FP64: 2e-15 of the density; FP32 deviations 2e-6)."""
import numpy as np
import pytest

from paper_1412_5170_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 2e-15), ("fp32", 2e-6)])
@pytest.mark.parametrize("nx,ny", [(1, 300001), (3, 100003), (8, 131072), (65599, 7), (1500007, 2), (1500007, 1)])
def test_start_at_rest(lbm, nx, ny, precision, tol):
    import torch
    rv, rl = lbm.maxwell(0.8)
    rho0 = rv + (rl - rv) * np.random.default_rng(nx).random((ny, nx))
    with lbm.Lattice(lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", precision)) as lat:
        d = torch.from_numpy(rho0).cuda()
        torch.cuda.synchronize()
        lat.init_density_dev(d)
        rho, _, _ = lat.read_moments()
    assert (np.abs(rho - rho0) / rho0).max() < tol


@pytest.mark.parametrize("nx,ny", [(1, 300001), (8, 131072), (1500007, 1)])
def test_preset(lbm, nx, ny):
    rv, rl = lbm.maxwell(0.8)
    want = synth.density_field(nx, ny, "droplet_array", rl, rv, 20.0, seed=11, noise_amp=1e-6, cell=97)
    with lbm.Lattice(lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", "fp64")) as lat:
        lat.init_preset("droplet_array", 20.0, seed=11, noise_amp=1e-6, cell=97)
        rho, _, _ = lat.read_moments()
    np.testing.assert_allclose(rho, want, rtol=0, atol=1e-15)
