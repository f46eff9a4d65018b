"""The moment fields alone (tiles; FP32 strips from 2^23 nodes) at shapes where
a tile or its ring can go wrong, against the moments of the populations that the
same lattice gives out: rho = sum f, and v = (j + F/2)/rho with psi and the force
evaluated here.

FP64: nine additions and the force's dozen operations, 1e-13 of the largest
|v| and 2e-15 of the density.  FP32: the element-wise bar of 2e-5 on the density,
1e-5 absolute on v (densities from 0.02: eight digits of the populations over
rho)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]


def moments(lbm, f, T, A, K):
    rho = f.sum(0)
    jx, jy = (sum(e[i] * f[a] for a, e in enumerate(E)) for i in (0, 1))
    t = T * lbm.tc()
    p = K * (rho * t * (1 + rho + rho ** 2 - rho ** 3) / (1 - rho) ** 3 - rho ** 2)
    psi = np.sqrt(2 * (rho / 3 - p))
    F = np.zeros((2,) + rho.shape)
    for a, (ex, ey) in enumerate(E[1:], 1):
        w = 1 / 3 if a < 5 else 1 / 12
        n = np.roll(psi, (-ey, -ex), axis=(0, 1))       # psi(x + e)
        phi = n * (A / 2 * n + (1 - A) * psi)
        F += w * np.array([ex * phi, ey * phi])
    return rho, (jx + F[0] / 2) / rho, (jy + F[1] / 2) / rho


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 331), (331, 1), (2, 97), (67, 3), (31, 257), (263, 129), (64, 64), (1023, 511), (20001, 3),
                                   (8, 40000), (4096, 2049)])
def test_moments(lbm, nx, ny, precision):
    rng = np.random.default_rng(nx + ny)
    rho0 = 0.02 + 0.28 * rng.random((ny, nx))
    f = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None] * rho0 * (1 + 0.05 * rng.random((9, ny, nx)))
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, "bgk", "guo", precision)
    with lbm.Lattice(p) as lat:
        lat.write_populations(f)
        got = lat.read_moments()
        again = lat.read_moments()
        f = lat.read_populations()
    assert all(np.array_equal(a, b) for a, b in zip(got, again))
    want = moments(lbm, f, 0.8, -0.304, 1.0)
    vmax = max(np.abs(want[1]).max(), np.abs(want[2]).max())
    assert (np.abs(got[0] - want[0]) / want[0]).max() < (2e-15 if precision == "fp64" else 2e-5)
    for g, w in zip(got[1:], want[1:]):
        assert np.abs(g - w).max() < (1e-13 * vmax + 1e-16 if precision == "fp64" else 1e-5)
