"""Six steps per launch over lists of two-species D2Q9 grids (a level's carried
rows in shared memory) and the default depth of a list by its size: the bits
of single-step launches."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu

# (8, 1): windows wrap several times; 52, 53: one strip exactly (64 - 2 * 6 columns) and one more column
SIZES = [(8, 1), (52, 30), (53, 7), (256, 24), (1200, 6), (416, 300)]


def _run(sizes, reactions, depth, steps):
    cfgs = [dict(lattice="D2Q9", nspecies=2, reaction=r, precision="fp32", nx=nx, ny=ny, tau=[0.8, 0.6 + 0.01 * j],
                 F=0.03, k=0.06, tb_depth=depth) for j, ((nx, ny), r) in enumerate(zip(sizes, reactions))]
    with B.Batch(cfgs) as b:
        for j, (nx, ny) in enumerate(sizes):
            rng = np.random.default_rng(j)
            b.init(j, np.stack([0.5 + 0.5 * rng.random((ny, nx)), 0.25 * rng.random((ny, nx))]))
        before = B.lb_rd_batch_get_time(b.b)[1]
        b.step(steps)
        launches = B.lb_rd_batch_get_time(b.b)[1] - before
        return [b.moments(j)[0] for j in range(len(sizes))], launches


@pytest.mark.parametrize("steps", [6, 13])
@pytest.mark.parametrize("mixed", [False, True], ids=["gray_scott", "mixed"])
@pytest.mark.parametrize("aligned", [True, False], ids=["nx4", "any_nx"])
def test_six_steps_equal_single_steps(aligned, mixed, steps):
    sizes = [(-(-nx // 4) * 4, ny) if aligned else (nx, ny) for nx, ny in SIZES]
    reactions = ["gray_scott", "none"] * 3 if mixed else ["gray_scott"] * 6
    want, _ = _run(sizes, reactions, 1, steps)
    got, _ = _run(sizes, reactions, 6, steps)
    for j, (w, g) in enumerate(zip(want, got)):
        np.testing.assert_array_equal(g, w, err_msg=str(sizes[j]))


@pytest.mark.parametrize("ny,launches", [(1535, 3), (1536, 2)])
def test_default_depth_of_a_list_by_its_sites(ny, launches):
    """Two grids of 512 x ny: 12 steps are 5 + 5 + 2 below 1.5 * 2^20 sites and 6 + 6 from there on."""
    want, _ = _run([(512, ny)] * 2, ["gray_scott"] * 2, 1, 12)
    got, n = _run([(512, ny)] * 2, ["gray_scott"] * 2, 0, 12)
    for w, g in zip(want, got):
        np.testing.assert_array_equal(g, w)
    assert n == launches
