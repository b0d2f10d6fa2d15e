"""The read-out's partial sums: one per block that fits the device, whatever the
grid, so that what a server holds from its start serves every request."""
import pytest

from paper_1007_3109_gb300 import binding as B


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_bf16dev"])
def test_partial_sums_do_not_grow_with_the_grid(precision):
    """What a handle holds beside its state and densities is the same for every grid."""
    def scratch(nx, ny):
        n = B.lb_rd_check_config(B.make_config("D2Q5", 1, nx, ny, [0.8], "none", precision=precision))
        site = {"fp64": 2 * 5 * 8 + 8, "fp32": 2 * 5 * 4 + 4, "fp32_bf16dev": 2 * (4 + 4 * 2) + 4}[precision]
        return n - site * nx * ny

    assert scratch(64, 64) == scratch(4096, 4128) == scratch(65504, 65535)


@pytest.mark.gpu
def test_server_reads_out_a_large_request():
    import numpy as np
    n = 4200  # 9 x 1050 tiles: more than fit the device at once
    rho0 = np.random.default_rng(0).random((1, n, n))
    kw = dict(lattice="D2Q5", nspecies=1, precision="fp32")
    with B.Server(8 << 30, **kw) as srv:
        rho, mass, _ = srv.result(srv.submit(rho0, 1, nx=n, ny=n, tau=[0.8], reaction="none", **kw))
    # the densities are floats; their sum in any order of FP64 additions
    assert abs(mass[0] - rho.sum()) <= n * n * 2.0 ** -53 * rho.sum()
