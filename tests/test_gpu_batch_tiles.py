"""The batched step on tiles (the automatic choice of small batches) against
the one-warp walk (asked for by set_tuning), every scheme, at shapes where
tiles and walk can disagree: the smallest width, single rows, sides that do
not divide into tiles, ragged last strips; and across a compaction, when
instances stop.

Both evaluate the same FP32 update per node: 2e-6 of the density after 40
steps (a tenth of the FP32 element-wise bar).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def instances(forc):
    A = 0.0 if forc == "li" else -0.304
    shapes = [(4, 1), (4, 37), (8, 127), (36, 5), (100, 33), (132, 130), (260, 36)]
    return [dict(nx=nx, ny=ny, kind="slab" if ny > 1 else "droplet", T_over_Tc=0.8, tau=0.8 + 0.05 * i, A=A, K=1.0,
                 size=max(1.5, ny / 4), seed=i) for i, (nx, ny) in enumerate(shapes)]


@pytest.mark.parametrize("coll,forc", [("mrt", "guo"), ("bgk", "guo"), ("bgk", "edm"), ("bgk", "sc"), ("bgk", "li")])
def test_tiles_match_walk(lbm, coll, forc):
    inst, out = instances(forc), []
    for walk in (False, True):
        with lbm.Batch(inst, collision=coll, forcing=forc, sigma=0.105 if forc == "li" else 0.0) as b:
            if walk:
                b.set_tuning(128, 3, 32)
            b.init()
            b.step(40)
            b.observe()
            state, code, steps, _ = b.results()
            assert (state == lbm.RUNNING).all() and (code == 0).all() and (steps == 40).all()
            out.append([b.read_density(i) for i in range(len(inst))])
    for x, y in zip(*out):
        assert (np.abs(x - y) / y).max() < 2e-6


def test_tiles_follow_the_running_instances(lbm):
    """Graph-captured intervals: a failing instance and three converging
    slabs leave the table at its compaction, and the last one runs on."""
    inst = [dict(nx=8, ny=64, kind="slab", T_over_Tc=0.85, tau=1.0, A=-0.304, K=1.0, size=16.0, seed=i, noise_amp=0.0)
            for i in range(3)]
    inst += [dict(nx=16, ny=16, kind="droplet", T_over_Tc=0.55, tau=0.51, A=0.9, K=1.0, size=5.0, seed=7),
             dict(nx=64, ny=64, kind="droplet", T_over_Tc=0.8, tau=1.0, A=-0.304, K=1.0, size=15.0, seed=8)]
    with lbm.Batch(inst) as b:
        b.init()
        b.run_to_steady(tol_coex=1e-6, check_every=200, max_steps=20000)
        state, code, steps, obs = b.results()
    assert state[3] == lbm.FAILED and code[3] in (lbm.E_NONFINITE, lbm.E_EOS_DOMAIN)
    assert (state[:3] == lbm.CONVERGED).all() and steps[3] < steps[:3].min() + 20000
    assert np.ptp(obs["rho_row_mid"][:3]) < 1e-6 and (obs["rho_row_mid"][:3] > 5 * obs["rho_row0"][:3]).all()


def test_large_batches_walk_tiles(lbm):
    """More than 3 * 2^20 nodes: chunks of tiles, against the one-warp walk."""
    inst = [dict(nx=512, ny=512, kind="droplet", T_over_Tc=0.8, tau=0.9, A=-0.304, K=1.0, size=100.0, seed=i) for i in range(12)]
    inst += [dict(nx=nx, ny=ny, kind="slab", T_over_Tc=0.75, tau=0.7, A=-0.304, K=0.5, size=ny / 4, seed=50 + ny)
             for nx, ny in ((4, 9), (36, 65), (516, 331))]
    out = []
    for walk in (False, True):
        with lbm.Batch(inst, collision="mrt") as b:
            if walk:
                b.set_tuning(128, 3, 32)
            b.init()
            b.step(20)
            out.append([b.read_density(i) for i in range(len(inst))])
    for x, y in zip(*out):
        assert (np.abs(x - y) / y).max() < 2e-6
