"""The K-step general kernels (one to four species, mass-action networks) give
the bits of single steps."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B
from paper_1007_3109_gb300 import inputs

pytestmark = pytest.mark.gpu

CUBIC2 = ([0.3, 0.02, 0.01, 0.05, 0.04], [(0, 3), (1, 0), (2, 1), (0, 0), (0, 2)],
          [(1, -1), (-1, 0), (0, 2), (1, 0), (0, -3)])
FULL16 = ([0.01 * (r + 1) for r in range(16)], [(r % 2, (r // 2) % 2, (r // 4) % 3) for r in range(16)],
          [((r % 3) - 1, ((r + 1) % 3) - 1, ((r + 2) % 3) - 1) for r in range(16)])
DECAY1 = ([0.02], [(1,)], [(-1,)])


@pytest.mark.parametrize("lat", ["D2Q9", "D2Q5"])
@pytest.mark.parametrize("S,net,taus", [(1, DECAY1, (0.9,)), (2, CUBIC2, (0.8, 0.65)), (3, FULL16, (0.7, 0.9, 1.4)),
                                        (3, None, (0.7, 0.9, 1.4)), (4, inputs.coupled_gs_network(), (0.8,) * 4)])
@pytest.mark.parametrize("nx,ny", [(4, 1), (28, 5), (56, 64), (228, 31)])
def test_general_depth_k_equals_single_steps(lat, S, net, taus, nx, ny):
    """Strips of 28 columns (one exactly, a ragged last one, a grid narrower
    than a window), every order 0 .. 3, the largest network and none at all;
    calls that end on K steps and on fewer."""
    rho0 = 0.1 + 0.5 * np.random.default_rng(nx + ny).random((S, ny, nx))
    kw = dict(reaction="none") if net is None else dict(reaction="mass_action", network=net)
    with B.Simulation(lat, S, nx, ny, list(taus), precision="fp32", track_mass=True, **kw) as sim:
        names = [B.lb_rd_handle_variant_name(sim.h, v) for v in range(B.lb_rd_handle_variant_count(sim.h))]
        deep = [v for v, name in enumerate(names) if B.variant_steps(name) > 1]
        assert {B.variant_steps(names[v]) for v in deep} == {2, 3}
        ref = {}
        for v in [0] + deep:
            sim.set_variant(v)
            sim.init(rho0)
            for n in (6, 7):
                sim.step(n)
                out = (*sim.moments(), sim.distributions())
                if v == 0:
                    ref[n] = out
                np.testing.assert_array_equal(out[0], ref[n][0], err_msg=names[v])
                np.testing.assert_array_equal(out[2], ref[n][2], err_msg=names[v])
                np.testing.assert_allclose(out[1], ref[n][1], rtol=1e-6)
