"""lb_rd_step captured into a caller's graph: calls of an even number of steps in
all leave the state in the copy where they found it, whatever the steps per
launch, so that every replay advances it."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B
from paper_1007_3109_gb300 import inputs

pytestmark = pytest.mark.gpu

GS = dict(nspecies=2, tau=[0.8, 0.65], reaction="gray_scott", F=0.04, k=0.06)
NET = dict(nspecies=4, tau=[0.8, 0.65] * 2, reaction="mass_action", network=inputs.coupled_gs_network())
CASES = [dict(GS, lattice="D2Q9", nx=512, ny=260, precision="fp32"), dict(GS, lattice="D2Q9", nx=511, ny=260, precision="fp32"),
         dict(GS, lattice="D2Q5", nx=512, ny=260, precision="fp32"),
         dict(GS, lattice="D2Q9", nx=512, ny=260, precision="fp32", track_mass=True),
         dict(GS, lattice="D2Q9", nx=512, ny=260, precision="fp32_bf16dev"),
         dict(NET, lattice="D2Q9", nx=300, ny=230, precision="fp32"),
         dict(GS, lattice="D2Q9", nx=512, ny=40, precision="fp32", tb_depth=3),
         dict(GS, lattice="D2Q9", nx=512, ny=40, precision="fp32", tb_depth=2),
         dict(GS, lattice="D2Q9", nx=90, ny=40, precision="fp64")]


@pytest.mark.parametrize("calls", [(2,), (10,), (26,), (30,), (1, 13), (7, 4, 9)])
@pytest.mark.parametrize("cfg", CASES, ids=lambda c: f"{c['lattice']}-{c['nspecies']}-{c['precision']}-{c['nx']}x{c['ny']}"
                         f"-mass{int(c.get('track_mass', False))}-K{c.get('tb_depth', 0)}")
def test_replays_advance_the_state(cfg, calls):
    import torch
    stream = torch.cuda.Stream()
    rho0 = 0.2 + 0.5 * np.random.default_rng(5).random((cfg["nspecies"], cfg["ny"], cfg["nx"]))
    with B.Simulation(**cfg, stream=stream.cuda_stream) as sim, B.Simulation(**cfg) as want:
        sim.init(rho0)
        want.init(rho0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for n in calls:
                sim.step(n)
        for _ in range(3):
            graph.replay()
            for n in calls:
                want.step(n)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(sim.distributions(), want.distributions())
        np.testing.assert_array_equal(sim.moments()[0], want.moments()[0])
