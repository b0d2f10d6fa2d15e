"""The FP64 step at the bottom of the number range: densities and reaction terms
of a few units of 2^-1074, whose product with the axis weight rounds to zero
while the one with the rest weight does not.  Every warp holds such values and
zeros only.  Bitwise against the oracle."""
import numpy as np
import pytest

import oracle as orc
from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu

UNIT = 5e-324  # 2^-1074


def _check(lat, taus, reaction, rho0, **kw):
    S, ny, nx = rho0.shape
    with B.Simulation(lat, S, nx, ny, taus, reaction, precision="fp64", **kw) as sim:
        sim.init(rho0)
        for steps in (1, 2, 3):
            want = orc.density(lat, orc.run(lat, taus, orc.Reaction(reaction, **kw), orc.init(lat, rho0), steps))
            np.testing.assert_array_equal(sim.step(1).moments()[0], want, err_msg=f"after {steps}")


@pytest.mark.parametrize("lat", ["D2Q9", "D2Q5"])
@pytest.mark.parametrize("n", range(1, 13))
@pytest.mark.parametrize("nx,ny", [(1, 1), (32, 4)])
def test_equal_densities(lat, n, nx, ny):
    for sign in (1.0, -1.0):
        _check(lat, [2.5], "none", np.full((1, ny, nx), sign * n * UNIT))


@pytest.mark.parametrize("lat", ["D2Q9", "D2Q5"])
@pytest.mark.parametrize("tau", [0.8, 1.0])
@pytest.mark.parametrize("seed", range(4))
def test_zeros_and_underflowing_densities(lat, tau, seed):
    _check(lat, [tau], "none", np.random.default_rng(seed).choice([0.0, 2.0, 3.0, 4.0], (1, 4, 32)) * UNIT)


@pytest.mark.parametrize("lat", ["D2Q9", "D2Q5"])
@pytest.mark.parametrize("n", range(1, 8))
def test_underflowing_reaction(lat, n):
    rho0 = np.zeros((2, 4, 32))
    rho0[0] = 1.0
    _check(lat, [0.8, 2.5], "linear", rho0, kappa=n * UNIT)
