"""The observables from walks of tiles against numpy on the moment fields the
same walk writes, at shapes where the walk or its reduction can go wrong: one
node, single rows and columns, one column more than a strip, ragged chunks,
odd sides (no strip walk), and the snapshot comparison.

The sums are FP64 (FP32: exact float pairs): 1e-12 of the mass.  Maxima are
exact up to the root's rounding in the compute type.
"""
import numpy as np
import pytest

from paper_1412_5170_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 300), (300, 1), (2, 3), (33, 8), (31, 257), (65, 41), (513, 67), (1030, 519)])
def test_stats_match_fields(lbm, nx, ny, precision):
    rv, rl = lbm.maxwell(0.8)
    rho0 = synth.density_field(nx, ny, "droplet", rl, rv, max(1.5, min(nx, ny) / 4), seed=9)
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", precision)
    eps = 1e-14 if precision == "fp64" else 3e-7
    with lbm.Lattice(p) as lat:
        lat.init_density(rho0)
        lat.step(3)
        assert lat.stats(snapshot=True)["max_dv"] == -1.0
        _, ux, uy = lat.read_moments()
        lat.step(2)
        a, b = lat.stats(snapshot=True), lat.stats()
        rho, vx, vy = lat.read_moments()
    assert a["status"] == 0 and b["max_dv"] == 0.0
    assert all(a[k] == b[k] for k in a if k != "max_dv")   # bit for bit from call to call
    assert a["mass"] == pytest.approx(rho.sum(), rel=1e-12)
    assert a["rho_row_mid"] == pytest.approx(rho[ny // 2].mean(), rel=1e-12)
    assert a["rho_row0"] == pytest.approx(rho[0].mean(), rel=1e-12)
    assert (a["rho_min"], a["rho_max"]) == (rho.min(), rho.max())
    assert (a["rho_center"], a["rho_corner"]) == (rho[ny // 2, nx // 2], rho[0, 0])
    assert a["max_v"] == pytest.approx(np.hypot(vx, vy).max(), rel=eps, abs=1e-300)
    assert a["max_dv"] == pytest.approx(np.hypot(vx - ux, vy - uy).max(), rel=10 * eps, abs=1e-12 if precision == "fp64" else 1e-7)
