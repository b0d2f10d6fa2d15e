"""Lists of grids on the two-column depth-K kernels: the rows of the list are
shared out among the blocks, cut where the shares end.  Every instance must
have the bits of single-step launches, whatever the cuts, the groups of strips
side by side and the grids' order."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu

LISTS = {
    "one strip, one row": [(8, 1)],
    "narrower than a window": [(16, 40), (16, 40), (24, 9)],
    "runs across groups": [(256, 24)] * 7 + [(112, 24)] * 3 + [(256, 24)],
    "one wide grid, few rows": [(1200, 6)],
    "more rows than workers": [(64, 700), (416, 300), (208, 515)],
    "uneven order": [(496, 33), (48, 260), (104, 1), (744, 12), (48, 260), (48, 12)],
    "many equal small grids": [(48, 20)] * 40,
}


def _run(sizes, lattice, precision, depth, steps):
    kw = dict(lattice=lattice, nspecies=2, reaction="gray_scott", precision=precision)
    cfgs = [dict(kw, nx=nx, ny=ny, tau=[0.8, 0.6 + 0.01 * j], F=0.03 + 1e-4 * j, k=0.06, tb_depth=depth)
            for j, (nx, ny) in enumerate(sizes)]
    out = []
    with B.Batch(cfgs) as b:
        for j, (nx, ny) in enumerate(sizes):
            rng = np.random.default_rng(100 + j)
            b.init(j, np.stack([0.5 + 0.5 * rng.random((ny, nx)), 0.25 * rng.random((ny, nx))]))
        b.step(steps)
        for j in range(len(sizes)):
            out.append(b.moments(j)[0])
    return out


@pytest.mark.parametrize("lattice,precision,depth", [("D2Q9", "fp32", 5), ("D2Q9", "fp32", 2), ("D2Q5", "fp32", 6),
                                                     ("D2Q9", "fp32_bf16dev", 4), ("D2Q5", "fp32_fp16dev", 5)])
@pytest.mark.parametrize("name", sorted(LISTS))
def test_list_equals_single_steps(name, lattice, precision, depth):
    sizes = LISTS[name]
    want = _run(sizes, lattice, precision, 1, 13)
    got = _run(sizes, lattice, precision, depth, 13)
    for j, (w, g) in enumerate(zip(want, got)):
        np.testing.assert_array_equal(g, w, err_msg=f"instance {j} of {name}")
    if precision == "fp32":  # the any-nx form
        odd = [(nx + 1, ny) for nx, ny in sizes]
        for j, (w, g) in enumerate(zip(_run(odd, lattice, precision, 1, 13), _run(odd, lattice, precision, depth, 13))):
            np.testing.assert_array_equal(g, w, err_msg=f"instance {j} of {name}, odd nx")
