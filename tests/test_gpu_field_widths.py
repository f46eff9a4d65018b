"""The built-in fields at the ends of the accepted interface widths.

Tolerances as in test_gpu_fields.py (FP64, 1e-15); the batch's FP32
deviations hold a density to 1e-6 of itself."""
import numpy as np
import pytest

from paper_1412_5170_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [1e-310, 5e-324, 1e-300, 1e300, float("inf")])
def test_extreme_widths(lbm, width):
    """Any positive width is accepted: the interface goes to a step (the node
    on it halfway) or to the mean everywhere."""
    rv, rl = lbm.maxwell(0.8)
    y, x = np.mgrid[0:8, 0:8]
    d = np.hypot(x - 4.0, y - 4.0) - 2.0
    with np.errstate(over="ignore"):
        want = rv + (rl - rv) * 0.5 * (1 - np.tanh(2 * d / width))
    with lbm.Lattice(lbm.make_params(8, 8, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", "fp64")) as lat:
        lat.init_preset("droplet", 2.0, width=width, noise_amp=0.0)
        rho, _, _ = lat.read_moments()
    np.testing.assert_allclose(rho, want, rtol=0, atol=1e-15)
    with lbm.Batch([dict(side=8, kind="droplet", T_over_Tc=0.8, tau=0.9, A=-0.304, K=1.0, size=2.0, width=width, noise_amp=0.0)]) as b:
        b.init()
        np.testing.assert_allclose(b.read_density(0), want, rtol=1e-6)
