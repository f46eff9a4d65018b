"""Steps at shapes that no other test reaches: walks of tiles on lattices of
one column and of fewer than eight rows (they need 2^17 nodes), one-warp strip
walks of a batch through graph-captured intervals, and a batch whose tile table
is rebuilt around its last running instance."""
import numpy as np
import pytest

import oracle
from paper_1412_5170_gb300 import synth

pytestmark = pytest.mark.gpu
MRT = dict(s_e=0.8, s_eps=0.8, s_q=1.1)


@pytest.mark.parametrize("coll,forc", [("mrt", "guo"), ("bgk", "edm")])
@pytest.mark.parametrize("nx,ny", [(1, 131101), (3, 43711), (131101, 1), (43711, 3), (18731, 7)])
def test_tile_walks_of_thin_lattices(lbm, nx, ny, coll, forc):
    """Against the oracle, at the FP32 element-wise bar of 2e-5 on the density."""
    rv, rl = lbm.maxwell(0.8)
    rho0 = synth.density_field(nx, ny, "slab" if ny > nx else "droplet_array", rl, rv, ny / 4 if ny > nx else 1.5, seed=5, cell=9)
    p = lbm.make_params(nx, ny, 0.8, 0.9, -0.304, 1.0, coll, forc, "fp32", **MRT)
    with lbm.Lattice(p) as lat:
        assert lat.config == 0
        lat.init_density(rho0)
        lat.step(8)
        f, st = lat.read_populations(), lat.stats()
    ref, ost = oracle.run(oracle.params(nx, ny, 0.8, 0.9, -0.304, 1.0, coll, forc, **MRT), oracle.init_rest(rho0), 8)
    assert ost == 0 and st["status"] == 0
    assert (np.abs(f.sum(0) - ref.sum(0)) / ref.sum(0)).max() < 2e-5


def slabs_and_a_failure():
    inst = [dict(nx=8, ny=64, kind="slab", T_over_Tc=0.85, tau=1.0, A=-0.304, K=1.0, size=16.0, seed=i, noise_amp=0.0) for i in range(3)]
    inst += [dict(nx=16, ny=16, kind="droplet", T_over_Tc=0.55, tau=0.51, A=0.9, K=1.0, size=5.0, seed=7),   # unstable
             dict(nx=160, ny=160, kind="droplet", T_over_Tc=0.8, tau=1.0, A=-0.304, K=1.0, size=40.0, seed=8)]
    return inst


@pytest.mark.parametrize("tuning", [None, (128, 3, 16, False), (128, 4, 32, False), (128, 2, 16, True)])
def test_intervals_and_compaction(lbm, tuning):
    """Tiles (the automatic choice) and one-warp walks: the failing instance
    and the slabs leave at a compaction, the droplet runs on after them and ends
    where the same lattice ends alone."""
    inst, steps_max = slabs_and_a_failure(), 6000
    with lbm.Batch(inst) as b:
        if tuning:
            b.set_tuning(*tuning)
        b.init()
        st, done = b.run_to_steady(tol_coex=2e-6, check_every=200, max_steps=steps_max)
        state, code, steps, _ = b.results()
        rho = b.read_density(4)
    assert state[3] == lbm.FAILED and code[3] in (lbm.E_NONFINITE, lbm.E_EOS_DOMAIN)
    assert (state[:3] == lbm.CONVERGED).all() and steps[3] < steps[:3].min() and steps[:3].max() < steps_max
    assert state[4] in (lbm.CONVERGED, lbm.RUNNING) and steps[4] == done > steps[:3].max()
    assert st == (lbm.OK if state[4] == lbm.CONVERGED else lbm.E_NOT_CONVERGED)
    with lbm.Batch(inst[4:]) as alone:
        if tuning:
            alone.set_tuning(*tuning)
        alone.init()
        alone.step(int(steps[4]))
        want = alone.read_density(0)
    # the same FP32 update of the same nodes: equal whatever else the batch held
    assert np.array_equal(rho, want)
