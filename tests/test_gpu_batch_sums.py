"""The sums of a batch's observables (mass, probe rows) are FP64 sums.

One 32 x 8 tile: eight additions down a column, five across, one each for the
nodes' reference and the fold of the tiles: sixteen roundings at most, so the
mass is within 16 * 2^-53 of the correctly rounded sum of the densities (a
row within ten).  Slabs whose deviations span 1e-12 to 0.3 make sums in less
than FP64 show: float pairs were off by up to 48 * 2^-53 here.  Ragged and
many-tile instances: one more rounding a tile."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("shapes", [[(32, 8)] * 400, [(4, 1), (4, 9), (28, 7), (36, 8), (260, 36), (8, 127), (64, 64)] * 20])
def test_sums_are_fp64(lbm, shapes):
    inst = [dict(nx=nx, ny=ny, kind="slab", T_over_Tc=0.8, tau=0.9, A=-0.304, K=1.0, size=ny / 4, width=1.0, rho_l=0.31, rho_v=0.0217,
                 noise_amp=1e-3, seed=i) for i, (nx, ny) in enumerate(shapes)]
    worst = [0.0, 0.0, 0.0]
    with lbm.Batch(inst) as b:
        b.init()
        b.observe()
        _, _, _, obs = b.results()
        for i, (nx, ny) in enumerate(shapes):
            rho = b.read_density(i)
            tiles = -(-nx // 32) * -(-ny // 8)
            for j, (got, rows, bar) in enumerate(((obs["mass"][i], rho, 16 + tiles), (obs["rho_row_mid"][i] * nx, rho[ny // 2], 11 + tiles),
                                                  (obs["rho_row0"][i] * nx, rho[0], 11 + tiles))):
                want = math.fsum(rows.ravel())
                worst[j] = max(worst[j], abs(got - want) / want / U / bar)
    assert max(worst) < 1, worst


def test_an_infinite_density_is_an_infinite_mass(lbm):
    inst = [dict(nx=32, ny=8, kind="slab", T_over_Tc=0.8, tau=0.9, A=-0.304, K=1.0, size=2.0, rho_l=rl, rho_v=0.0217, noise_amp=0.0)
            for rl in (0.31, np.inf)]
    with lbm.Batch(inst) as b:
        b.init()
        b.observe()
        state, code, _, obs = b.results()
    assert state[1] == lbm.FAILED and obs["mass"][1] == np.inf and state[0] == lbm.RUNNING and np.isfinite(obs["mass"][0])
