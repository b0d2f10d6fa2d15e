"""lb_rd_batch_step captured into a caller's graph before the batch has run: full
launches and single steps need nothing that is not there since the batch was made.
The replay has the bits of the same call without a capture, and a call of an even
number of steps can be replayed again."""
import numpy as np
import pytest

from paper_1007_3109_gb300 import binding as B

pytestmark = pytest.mark.gpu

SIZES = [(64, 40), (48, 17)]


def _batch(depth, precision, stream=None):
    b = B.Batch([dict(lattice="D2Q9", nspecies=2, nx=nx, ny=ny, tau=[0.8, 0.65], reaction="gray_scott", F=0.04, k=0.06,
                      precision=precision, tb_depth=depth, stream=stream) for nx, ny in SIZES])
    for j, (nx, ny) in enumerate(SIZES):
        b.init(j, 0.2 + 0.5 * np.random.default_rng(j).random((2, ny, nx)))
    return b


@pytest.mark.parametrize("depth,precision,steps", [(5, "fp32", 5), (5, "fp32", 6), (5, "fp32", 11), (6, "fp32", 13),
                                                   (4, "fp32", 9), (4, "fp32_bf16dev", 9)])
def test_first_call_captured(depth, precision, steps):
    import torch
    stream = torch.cuda.Stream()
    with _batch(depth, precision, stream.cuda_stream) as b, _batch(depth, precision) as want:
        want.step(steps)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            b.step(steps)
        graph.replay()
        torch.cuda.synchronize()
        assert b.time == want.time == steps
        for j in range(len(SIZES)):
            np.testing.assert_array_equal(b.moments(j)[0], want.moments(j)[0])
        # outside a capture the same call goes on from there
        b.step(steps)
        want.step(steps)
        for j in range(len(SIZES)):
            np.testing.assert_array_equal(b.moments(j)[0], want.moments(j)[0])


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("depth,precision", [(6, "fp32"), (5, "fp32"), (4, "fp32"), (4, "fp32_bf16dev")])
@pytest.mark.parametrize("steps", [2, 4, 6, 10, 12, 20, 30])
def test_replays_advance_the_batch(depth, precision, steps, warm):
    import torch
    stream = torch.cuda.Stream()
    with _batch(depth, precision, stream.cuda_stream) as b, _batch(1, precision) as want:
        if warm:  # the depths of the call's last steps are planned
            b.step(steps)
            want.step(steps)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            b.step(steps)
        for _ in range(3):
            graph.replay()
            want.step(steps)
        torch.cuda.synchronize()
        for j in range(len(SIZES)):
            np.testing.assert_array_equal(b.moments(j)[0], want.moments(j)[0], err_msg=f"instance {j}")


def test_default_depth_of_a_large_batch_replays():
    """Seven grids of 512^2: the default depth, 20 steps as before it was six."""
    import torch
    stream = torch.cuda.Stream()

    def make(depth, st=None):
        b = B.Batch([dict(lattice="D2Q9", nspecies=2, nx=512, ny=512, tau=[0.8, 0.65], reaction="gray_scott", F=0.04,
                          k=0.06, precision="fp32", tb_depth=depth, stream=st)] * 7)
        for j in range(7):
            b.init(j, 0.2 + 0.5 * np.random.default_rng(j).random((2, 512, 512)))
        return b

    with make(0, stream.cuda_stream) as b, make(1) as want:
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            b.step(20)
        for _ in range(2):
            graph.replay()
            want.step(20)
        torch.cuda.synchronize()
        for j in range(7):
            np.testing.assert_array_equal(b.moments(j)[0], want.moments(j)[0], err_msg=f"instance {j}")
