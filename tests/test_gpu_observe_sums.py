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


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(65537, 1), (20001, 3), (9601, 17), (40000, 2), (131072, 1), (4097, 259)])
def test_more_pieces_than_ctas(lbm, nx, ny, precision):
    """Wide flat lattices: a CTA observes several pieces and reduces once
    (and flat ones of strips' widths go to the strips).  Sums are FP64: 1e-12
    of the mass; maxima exact up to the root's rounding."""
    rv, rl = lbm.maxwell(0.8)
    rho0 = rv + (rl - rv) * np.random.default_rng(ny).random((ny, nx))
    eps = 1e-14 if precision == "fp64" else 3e-7
    with lbm.Lattice(lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", precision)) as lat:
        lat.init_density(rho0)
        lat.stats(snapshot=True)
        _, ux, uy = lat.read_moments()
        lat.step(1)
        a, b = lat.stats(snapshot=True), lat.stats()
        rho, vx, vy = lat.read_moments()
    assert b["max_dv"] == 0.0 and all(a[k] == b[k] for k in a if k != "max_dv")   # bit for bit from call to call
    assert a["mass"] == pytest.approx(rho.sum(), rel=1e-12)
    assert a["rho_row_mid"] == pytest.approx(rho[ny // 2].mean(), rel=1e-12)
    assert a["rho_row0"] == pytest.approx(rho[0].mean(), rel=1e-12)
    assert (a["rho_min"], a["rho_max"]) == (rho.min(), rho.max())
    assert (a["rho_center"], a["rho_corner"]) == (rho[ny // 2, nx // 2], rho[0, 0])
    assert a["max_v"] == pytest.approx(np.hypot(vx, vy).max(), rel=eps)
    assert a["max_dv"] == pytest.approx(np.hypot(vx - ux, vy - uy).max(), rel=10 * eps)
