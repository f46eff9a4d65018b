"""The strip observation of large FP32 lattices (3 * 2^20 nodes and more at
widths that 512-column strips cover) against numpy on the moment fields:
several calls in a row (the last-CTA counter must be ready again), ragged last
strips, row chunks of unequal height, the snapshot stored and compared, and
the call without a snapshot.

The sums are exact float pairs per thread and FP64 beyond: 1e-12 of the mass;
a probe row is 1e-12 too.  Maxima are exact up to the root's rounding in
FP32 (3e-7), the change of v to one more subtraction (3e-6)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1540, 2053), (516, 9001), (2044, 1601), (4100, 1031), (512, 6151), (3072, 1024)])
def test_stats_match_fields(lbm, nx, ny):
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "mrt", "guo", "fp32", s_e=0.8, s_eps=0.8, s_q=1.1)
    with lbm.Lattice(p) as lat:
        lat.init_preset("droplet_array", min(nx, ny) / 8, cell=min(nx, ny) // 3, seed=6, noise_amp=1e-4)
        assert lat.stats(snapshot=True)["max_dv"] == -1.0
        _, ux, uy = lat.read_moments()
        for k in range(3):
            lat.step(2)
            a = lat.stats(snapshot=True)
            rho, vx, vy = lat.read_moments()
            again = lat.stats()
            assert again["max_dv"] == 0.0 and all(a[f] == again[f] for f in a if f != "max_dv")
            assert a["status"] == 0 and a["steps"] == 2 * (k + 1)
            assert a["mass"] == pytest.approx(rho.sum(), rel=1e-12)
            assert a["rho_row_mid"] == pytest.approx(rho[ny // 2].mean(), rel=1e-12)
            assert a["rho_row0"] == pytest.approx(rho[0].mean(), rel=1e-12)
            assert (a["rho_min"], a["rho_max"]) == (rho.min(), rho.max())
            assert (a["rho_center"], a["rho_corner"]) == (rho[ny // 2, nx // 2], rho[0, 0])
            assert a["max_v"] == pytest.approx(np.hypot(vx, vy).max(), rel=3e-7)
            assert a["max_dv"] == pytest.approx(np.hypot(vx - ux, vy - uy).max(), rel=3e-6)
            ux, uy = vx, vy


def test_fields_match_the_walk_of_tiles(lbm):
    """The same state on two widths that differ in how it is observed: a
    lattice of strips' width against itself shifted into the walk of tiles
    (FP64 moments of the same FP32 populations), node by node."""
    nx, ny = 1540, 2053
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "mrt", "guo", "fp32", s_e=0.8, s_eps=0.8, s_q=1.1)
    with lbm.Lattice(p) as lat:
        lat.init_preset("droplet_array", 200.0, cell=600, seed=6)
        lat.step(3)
        f, (rho, vx, vy) = lat.read_populations(), lat.read_moments()
    # a tall copy: rows repeated until the periodic neighbours of the kept rows are the same
    rows = slice(900, 1100)
    q = lbm.make_params(nx, 204, 0.8, 0.9, -0.304, 1.0, "mrt", "guo", "fp32", s_e=0.8, s_eps=0.8, s_q=1.1)
    with lbm.Lattice(q) as part:                     # 314 160 nodes: walks of tiles
        part.write_populations(np.ascontiguousarray(f[:, 898:1102]))
        prho, pvx, pvy = part.read_moments()
    assert np.abs(prho[2:-2] - rho[rows]).max() < 1e-6 * rho.max()
    assert max(np.abs(pvx[2:-2] - vx[rows]).max(), np.abs(pvy[2:-2] - vy[rows]).max()) < 2e-6
