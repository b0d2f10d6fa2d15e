"""Calls of every length on batches of K steps per launch: the steps left after
the full launches are shared out over two launches.  The bits, the batch time
and the densities are those of single steps, and no call takes more launches
than ceil(steps / K)."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _batch(lattice, precision, depth, sizes):
    return B.Batch([dict(lattice=lattice, nspecies=2, reaction="gray_scott", precision=precision, nx=nx, ny=ny,
                         tau=[0.8, 0.65], F=0.03, k=0.06, tb_depth=depth) for nx, ny in sizes])


@pytest.mark.parametrize("lattice,precision,depth", [("D2Q9", "fp32", 6), ("D2Q9", "fp32", 5), ("D2Q5", "fp32", 3),
                                                     ("D2Q9", "fp32", 8), ("D2Q9", "fp32_bf16dev", 4)])
def test_calls_of_every_length(lattice, precision, depth):
    sizes = [(48, 20), (64, 9)]
    rng = np.random.default_rng(5)
    rho = [np.stack([0.5 + 0.5 * rng.random((ny, nx)), 0.25 * rng.random((ny, nx))]) for nx, ny in sizes]
    with _batch(lattice, precision, 1, sizes) as one, _batch(lattice, precision, depth, sizes) as many:
        for b in (one, many):
            b.set_graph(2 * depth)
            for j, r in enumerate(rho):
                b.init(j, r)
        for steps in range(1, 4 * depth + 2):
            one.step(steps)
            before = B.lb_rd_batch_get_time(many.b)[1]
            many.step(steps)
            assert many.time == one.time
            assert B.lb_rd_batch_get_time(many.b)[1] - before == -(-steps // depth)
            for j in range(len(sizes)):
                np.testing.assert_array_equal(many.moments(j)[0], one.moments(j)[0], err_msg=f"{steps} steps")
