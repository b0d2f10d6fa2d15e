"""Untuned handles: above 65536 sites several steps per launch, chosen by size,
with the bits of one step per launch (densities, populations and the tracked
mass)."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B
from paper_1007_3109_gb300 import inputs

pytestmark = pytest.mark.gpu

NET3 = ([0.3, 0.05, 0.02, 0.01], [(1, 1, 0), (0, 0, 1), (0, 0, 1), (0, 0, 0)],
        [(-1, -1, 1), (1, 1, -1), (0, 0, -1), (1, 0, 0)])
GS = dict(nspecies=2, tau=[0.8, 0.65], reaction="gray_scott", F=0.04, k=0.06)
LIN = dict(nspecies=1, tau=[0.9], reaction="linear", kappa=1e-3)

# each of the rule's choices, on both sides of its lines
GRIDS = [(GS, "D2Q9", "fp32", 300, 219), (GS, "D2Q9", "fp32", 1540, 1024), (GS, "D2Q9", "fp32", 257, 256),
         (GS, "D2Q9", "fp32", 769, 513), (GS, "D2Q5", "fp32", 512, 130), (GS, "D2Q5", "fp32", 511, 131),
         (LIN, "D2Q9", "fp32", 264, 250), (LIN, "D2Q5", "fp32", 65532, 2), (GS, "D2Q9", "fp32_bf16dev", 264, 260),
         (GS, "D2Q9", "fp32_fp16dev", 268, 250), (LIN, "D2Q5", "fp32_bf16dev", 1028, 2048),
         (dict(nspecies=4, tau=[0.8, 0.65] * 2, reaction="mass_action", network=inputs.coupled_gs_network()), "D2Q9",
          "fp32", 260, 256),
         (dict(nspecies=3, tau=[0.7, 0.9, 1.4], reaction="mass_action", network=NET3), "D2Q5", "fp32", 300, 300)]


@pytest.mark.parametrize("mass", [False, True])
@pytest.mark.parametrize("phys,lat,prec,nx,ny", GRIDS,
                         ids=[f"{g[1]}-{g[0]['nspecies']}-{g[2]}-{g[3]}x{g[4]}" for g in GRIDS])
def test_untuned_handle_equals_one_step_per_launch(phys, lat, prec, nx, ny, mass):
    S = phys["nspecies"]
    rho0 = 0.2 + 0.5 * np.random.default_rng(nx + ny).random((S, ny, nx))
    kw = dict(lattice=lat, nx=nx, ny=ny, precision=prec, track_mass=mass, **phys)
    with B.Simulation(**kw) as sim, B.Simulation(**kw) as ref:
        assert B.variant_steps(B.lb_rd_handle_variant_name(sim.h, B.lb_rd_get_variant(sim.h))) > 1
        ref.set_variant(0)
        sim.init(rho0)
        ref.init(rho0)
        for n in (1, 2, 13, 7):
            l0 = B.lb_rd_launch_count(sim.h)
            sim.step(n)
            ref.step(n)
            assert n < 7 or B.lb_rd_launch_count(sim.h) - l0 < n
            rho, m = sim.moments()
            want, mw = ref.moments()
            np.testing.assert_array_equal(rho, want, err_msg=f"after {n}")
            np.testing.assert_array_equal(m, mw, err_msg=f"mass after {n}")
        np.testing.assert_array_equal(sim.distributions(), ref.distributions())
        assert sim.time == ref.time == 23


@pytest.mark.parametrize("kw", [dict(GS, lattice="D2Q9", nx=256, ny=256), dict(GS, nx=300, ny=300, precision="fp64"),
                                dict(GS, nx=300, ny=300, inplace=True), dict(GS, nx=300, ny=300, tb_depth=1)])
def test_where_one_step_per_launch_stays(kw):
    with B.Simulation(**kw) as sim:
        sim.init(np.full((2, kw["ny"], kw["nx"]), 0.5))
        l0 = B.lb_rd_launch_count(sim.h)
        sim.step(11)
        assert B.lb_rd_launch_count(sim.h) - l0 == 11
