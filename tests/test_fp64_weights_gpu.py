"""The FP64 step forms w_i rho from one product and powers of two where that is
the rounded product; densities whose products are subnormal, zero or overflow
take the products one by one.  Bitwise against the oracle for densities of every
magnitude, in single grids and in a batch of grids of any width."""
import numpy as np
import pytest

import oracle as orc
from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _rho0(S, ny, nx, seed, lo, hi):
    rng = np.random.default_rng(seed)
    r = 10.0 ** rng.uniform(lo, hi, (S, ny, nx)) * rng.choice([-1.0, 1.0], (S, ny, nx))
    r[rng.random((S, ny, nx)) < 0.1] = 0.0
    return r


@pytest.mark.parametrize("lat", ["D2Q9", "D2Q5"])
@pytest.mark.parametrize("S,taus", [(1, [1.0]), (2, [0.8, 1.0])])
@pytest.mark.parametrize("lo,hi", [(-323.0, -300.0), (-2.0, 2.0), (290.0, 308.0), (-320.0, 300.0)])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 31), (100, 7), (129, 3)])
def test_every_magnitude_bitwise(lat, S, taus, lo, hi, nx, ny):
    rho0 = _rho0(S, ny, nx, nx + ny, lo, hi)
    with np.errstate(all="ignore"):
        want = orc.density(lat, orc.run(lat, taus, orc.Reaction("linear", kappa=0.01), orc.init(lat, rho0), 4))
    with B.Simulation(lat, S, nx, ny, taus, "linear", kappa=0.01, precision="fp64") as sim:
        sim.init(rho0).step(4)
        np.testing.assert_array_equal(sim.moments()[0], want)


def test_batch_of_uneven_grids_bitwise():
    sizes = [(100, 100), (1, 5), (31, 33), (257, 4), (128, 1), (50, 77)]
    cfgs = [dict(lattice="D2Q9", nspecies=2, nx=nx, ny=ny, tau=[0.8, 0.65], reaction="gray_scott", F=0.03 + 0.01 * j,
                 k=0.06, precision="fp64") for j, (nx, ny) in enumerate(sizes)]
    with B.Batch(cfgs) as b:
        for j, (nx, ny) in enumerate(sizes):
            b.init(j, 0.2 + 0.5 * np.random.default_rng(j).random((2, ny, nx)))
        b.step(9)
        for j, (nx, ny) in enumerate(sizes):
            rho0 = 0.2 + 0.5 * np.random.default_rng(j).random((2, ny, nx))
            reac = orc.Reaction("gray_scott", F=0.03 + 0.01 * j, k=0.06)
            want = orc.density("D2Q9", orc.run("D2Q9", [0.8, 0.65], reac, orc.init("D2Q9", rho0), 9))
            np.testing.assert_array_equal(b.moments(j)[0], want)
