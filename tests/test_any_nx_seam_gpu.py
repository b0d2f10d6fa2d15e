"""The any-nx two-column kernels stage the chunks at the periodic seam column by
column: every remainder of nx, last strips of every width and grids narrower than
a staged row have the bits of single steps."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat", ["D2Q9", "D2Q5"])
@pytest.mark.parametrize("nx", [5, 17, 53, 57, 58, 61, 62, 63, 65, 66, 67, 69, 70, 71, 103, 105, 110, 155, 157, 163, 209])
def test_seam_chunks(lat, nx):
    ny = 9
    rng = np.random.default_rng(nx)
    rho0 = np.stack([0.5 + 0.5 * rng.random((ny, nx)), 0.25 * rng.random((ny, nx))])
    names = [B.lb_rd_variant_name("fp32", v) for v in range(B.lb_rd_variant_count("fp32"))]
    kw = dict(tau=[0.8, 0.65], reaction="gray_scott", F=0.04, k=0.06, precision="fp32")
    with B.Simulation(lat, 2, nx, ny, **kw) as sim:
        sim.set_variant(0)
        want = sim.init(rho0).step(12).distributions()
        any_nx = [v for v, n in enumerate(names) if n.startswith("deep") and "a_" in n]
        assert len(any_nx) >= 4
        for v in any_nx:
            sim.set_variant(v)
            got = sim.init(rho0).step(12).distributions()
            np.testing.assert_array_equal(got, want, err_msg=names[v])
