"""The fused read-out (densities to FP64 and their sum in one pass): exact
conversion of every kind of float, odd and narrow rows, unaligned output
buffers, and each output alone."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("nx,ny", [(1, 1), (63, 5), (64, 33), (66, 4), (513, 9), (1030, 130)])
def test_readout_outputs_agree(precision, S, nx, ny):
    import torch
    rho0 = 0.5 + np.random.default_rng(nx).random((S, ny, nx))
    with B.Simulation("D2Q9", S, nx, ny, [0.8, 0.65][:S], "none", precision=precision) as sim:
        sim.init(rho0)
        rho, mass = sim.moments()
        pitch, dt = (nx + 31) // 32 * 32, np.float32 if precision == "fp32" else np.float64
        cache = np.frombuffer(sim.save(), dt)[-S * ny * pitch:].reshape(S, ny, pitch)  # a checkpoint ends on the cache
        np.testing.assert_array_equal(rho, cache[:, :, :nx].astype(np.float64))
        np.testing.assert_allclose(mass, rho.sum(axis=(1, 2)), rtol=1e-14)
        np.testing.assert_array_equal(sim.mass(), mass)
        # device buffers, the densities at an odd multiple of 8 bytes
        n = S * ny * nx
        buf = torch.zeros(n + 2, dtype=torch.float64, device="cuda")
        m = torch.zeros(S, dtype=torch.float64, device="cuda")
        B.lb_rd_moments(sim.h, buf[1:n + 1], m)
        np.testing.assert_array_equal(buf[1:n + 1].cpu().numpy().reshape(rho.shape), rho)
        np.testing.assert_array_equal(m.cpu().numpy(), mass)
        assert buf[0] == 0 and buf[n + 1] == 0
        f = torch.zeros(9 * n + 2, dtype=torch.float64, device="cuda")
        B.lb_rd_get_distributions(sim.h, f[1:9 * n + 1])
        np.testing.assert_array_equal(f[1:9 * n + 1].cpu().numpy().reshape(S, 9, ny, nx), sim.distributions())
        assert f[0] == 0 and f[9 * n + 1] == 0


def test_special_values_convert_exactly():
    """Zeros, subnormals, the largest and smallest normals, infinities and NaN in
    the density cache (through a checkpoint, whose last part is the cache)."""
    nx, ny = 40, 3
    with B.Simulation("D2Q9", 1, nx, ny, [0.8], "none", precision="fp32") as sim:
        sim.init(np.ones((1, ny, nx)))
        blob = sim.save()
        cache = np.frombuffer(blob, np.float32)[-ny * 64:].reshape(ny, 64)  # row pitch 64
        vals = np.array([0.0, -0.0, 1e-45, -1e-45, 1.1754942e-38, 1.17549435e-38, -1.17549435e-38, 3.4028235e38,
                         -3.4028235e38, np.inf, -np.inf, np.nan, 1.0, -1.0, 1.0000001, 16777217.0], np.float32)
        cache[0, :16] = vals
        cache[2, 23:39] = vals
        sim.restore(blob)
        rho = np.empty((1, ny, nx))
        B.lb_rd_moments(sim.h, rho, None)
        want = vals.astype(np.float64)
        for got in (rho[0, 0, :16], rho[0, 2, 23:39]):
            np.testing.assert_array_equal(got, want)
            assert np.array_equal(np.signbit(got[:11]), np.signbit(want[:11]))


def test_batch_readout_to_device():
    import torch
    cfg = dict(lattice="D2Q9", nspecies=2, nx=70, ny=31, tau=[0.8, 0.65], reaction="gray_scott", F=0.04, k=0.06)
    with B.Batch([cfg, dict(cfg, nx=130)]) as b:
        for j, nx in enumerate((70, 130)):
            b.init(j, 0.2 + 0.5 * np.random.default_rng(j).random((2, 31, nx)))
        b.step(9)
        for j, nx in enumerate((70, 130)):
            rho, mass = b.moments(j)
            r = torch.zeros((2, 31, nx), dtype=torch.float64, device="cuda")
            m = torch.zeros(2, dtype=torch.float64, device="cuda")
            B.lb_rd_batch_moments(b.b, j, r, m)
            np.testing.assert_array_equal(r.cpu().numpy(), rho)
            np.testing.assert_array_equal(m.cpu().numpy(), mass)
            np.testing.assert_allclose(mass, rho.sum(axis=(1, 2)), rtol=1e-14)
