"""lb_rd_batch_step captured into a caller's graph before the batch has run: full
launches and a single step need nothing that is not there since the batch was
made, so calls of q K and q K + 1 steps can be captured.  The replay has the bits
of the same call without a capture."""
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
