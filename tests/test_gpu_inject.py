"""lbm_inject_stage_timeout where a lattice steps on the generic kernel."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("choose", [lambda lat: setattr(lat, "variant", 0), lambda lat: setattr(lat, "config", 0)])
def test_a_caller_who_then_chooses_the_generic_kernel_gets_it(lbm, choose):
    """The generic kernel stages nothing, so a step that the caller put on it
    after the injection runs it and cannot time out."""
    with lbm.Lattice(lbm.make_params(1536, 1536, 0.8, 0.9, -0.304, 1.0, "mrt", "guo", "fp32", s_e=0.8, s_eps=0.8, s_q=1.1)) as lat:
        assert lat.config == 0
        lat.init_preset("droplet", 100.0)
        lat.inject_stage_timeout()
        choose(lat)
        lat.step(1)
        assert lat.stats()["status"] == 0
        lat.variant = -1
        lat.step(1)
        assert lat.stats()["status"] == 0      # the injection was for one step
