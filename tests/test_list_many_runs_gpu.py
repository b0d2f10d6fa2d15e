"""Lists of many different grids on the two-column kernels: a worker's place in
the list is found by bisection over the runs of equal grids.  The bits are those
of single steps, and a list of many runs takes about as long as the same grids
sorted into a few."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu

LISTS = {
    "two runs": [(64, 30)] * 3 + [(48, 17)],
    "three runs, the last one grid": [(32, 9)] * 5 + [(64, 40)] * 2 + [(24, 50)],
    "all different": [(40 + 8 * (j % 9), 20 + j) for j in range(65)],
    "alternating": [(32 + 8 * (j % 3), 12) for j in range(200)],
    "more rows than workers": [(64 + 8 * (j % 5), 300 + j) for j in range(33)],
}


def _batch(sizes, lattice, precision, depth):
    cfgs = [dict(lattice=lattice, nspecies=1, nx=nx, ny=ny, tau=[0.6 + 0.003 * j], reaction="linear", kappa=1e-3,
                 precision=precision, tb_depth=depth) for j, (nx, ny) in enumerate(sizes)]
    b = B.Batch(cfgs)
    for j, (nx, ny) in enumerate(sizes):
        b.init(j, 0.5 + 0.5 * np.random.default_rng(j).random((1, ny, nx)))
    return b


@pytest.mark.parametrize("lattice,precision,depth", [("D2Q9", "fp32", 5), ("D2Q5", "fp32", 6),
                                                     ("D2Q9", "fp32_bf16dev", 4)])
@pytest.mark.parametrize("name", sorted(LISTS))
def test_bits_of_single_steps(name, lattice, precision, depth):
    sizes = LISTS[name]
    with _batch(sizes, lattice, precision, 1) as one, _batch(sizes, lattice, precision, depth) as many:
        one.step(2 * depth + 1)
        many.step(2 * depth + 1)
        for j in range(len(sizes)):
            np.testing.assert_array_equal(many.moments(j)[0], one.moments(j)[0], err_msg=f"instance {j}")


def test_many_runs_take_no_longer_than_few():
    import torch

    def us(sizes):
        with _batch(sizes, "D2Q9", "fp32", 5) as b:
            b.step(60)
            times = []
            for _ in range(7):
                torch.cuda.synchronize()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                b.step(60)
                e1.record()
                torch.cuda.synchronize()
                times.append(e0.elapsed_time(e1) * 1e3)
            return min(times)

    sizes = [(32 + 8 * (j % 7), 40) for j in range(300)]
    assert us(sizes) < 1.3 * us(sorted(sizes))
