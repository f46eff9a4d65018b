"""The built-in initial fields, evaluated on the device, against the seeded
generator of the tests (numpy, FP64).

Tolerance (absolute, densities below 0.31): the nine-term population sum of
the moment read rounds nine times (3e-16), tanh is good to 2 ulp, and its
argument z <= 20 carries three roundings damped by sech^2 (z sech^2 z < 0.45):
below 1e-15 together.
"""
import numpy as np
import pytest

from paper_1412_5170_gb300 import synth

pytestmark = pytest.mark.gpu


# nodes beyond ten widths of the interface skip tanh; odd sides and cells move
# the centre between nodes; the widest interface never saturates
@pytest.mark.parametrize("kind", ["slab", "droplet", "bubble", "droplet_array"])
@pytest.mark.parametrize("nx,ny,size,width,cell,noise", [(1, 7, 2.0, 1.0, 3, 0.0), (5, 1, 1.5, 4.0, 2, 1e-6),
                                                         (257, 67, 20.25, 0.3, 33, 1e-5), (64, 301, 14.0, 400.0, 64, 1e-6)])
def test_preset_fields(lbm, kind, nx, ny, size, width, cell, noise):
    rv, rl = lbm.maxwell(0.8)
    want = synth.density_field(nx, ny, kind, rl, rv, size, width=width, seed=2 ** 63 + 5, noise_amp=noise, cell=cell)
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", "fp64")
    with lbm.Lattice(p) as lat:
        lat.init_preset(kind, size, width=width, seed=2 ** 63 + 5, noise_amp=noise, cell=cell)
        rho, _, _ = lat.read_moments()
    np.testing.assert_allclose(rho, want, rtol=0, atol=1e-15)
