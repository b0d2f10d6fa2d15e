"""Launch variants keep their index: a program that stored one gets the kernel it
chose, of as many steps per launch."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B
from paper_1007_3109_gb300 import inputs

pytestmark = pytest.mark.gpu

GENERAL = ["general_1site", "general_2site", "general_4site", "general_2site_minb3", "general_2pass_minb8",
           "general_2pass_minb10"]


def test_general_one_step_variants():
    net = inputs.coupled_gs_network()
    rho0 = 0.2 + 0.5 * np.random.default_rng(3).random((4, 20, 64))
    with B.Simulation("D2Q9", 4, 64, 20, [0.8, 0.65] * 2, "mass_action", network=net, precision="fp32") as sim:
        want = None
        for v, name in enumerate(GENERAL):
            assert B.lb_rd_handle_variant_name(sim.h, v) == name
            sim.set_variant(v)
            sim.init(rho0)
            before = B.lb_rd_launch_count(sim.h)
            sim.step(5)
            assert B.lb_rd_launch_count(sim.h) - before == 5
            rho = sim.moments()[0]
            want = rho if want is None else want
            np.testing.assert_array_equal(rho, want, err_msg=name)
