"""A chain of step launches, which overlap their starts, takes no longer than
the same launches one after the other (with an event between any two): the next
launch's blocks must not crowd onto a few of the SMs while this one runs."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,S,nx,ny", [("D2Q5", 2, 512, 160), ("D2Q9", 2, 137, 400), ("D2Q9", 1, 137, 837),
                                         ("D2Q5", 1, 512, 256), ("D2Q9", 2, 512, 512)])
def test_chain_against_single_launches_fp64(lat, S, nx, ny):
    import torch
    kw = dict(reaction="gray_scott", F=0.04, k=0.06) if S == 2 else dict(reaction="linear", kappa=0.01)
    with B.Simulation(lat, S, nx, ny, [0.8, 0.65][:S], precision="fp64", **kw) as sim:
        sim.init(0.2 + 0.5 * np.random.default_rng(1).random((S, ny, nx))).step(50)
        chain, single = [], []
        for _ in range(7):
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            sim.step(50)
            e1.record()
            torch.cuda.synchronize()
            chain.append(e0.elapsed_time(e1))
            B.lb_rd_set_timing(sim.h, True)
            sim.step(50)
            single.append(B.lb_rd_kernel_time(sim.h)[0])
            B.lb_rd_set_timing(sim.h, False)
        assert min(chain) < 1.1 * min(single), (min(chain), min(single))
