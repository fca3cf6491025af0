"""Whole-layer chains on two, three and four lanes (on three and four two CTAs share an SM): the same bits as one call after the other."""
import pytest
import torch

from paper_2203_12533_b200 import inputs
from tests.test_gpu_layer import run_chain_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


# the fewest tokens, K ranges of two to sixteen blocks, several key blocks, the most tokens with two CTAs an SM, and so many that the chain takes two lanes
@pytest.mark.parametrize("F,S,B,M", [(128, 128, 1, 4), (1024, 128, 2, 3), (1024, 128, 2, 5), (640, 384, 1, 4), (1408, 128, 3, 4), (1024, 512, 1, 4), (1024, 128, 4, 3), (1024, 640, 1, 4)])
def test_same_bits(pw, F, S, B, M):
    w = inputs.Workload("lanes", 256, 4, 64, F, S, B, sigma_w=0.05)
    for schedule, recompute in ((pw.SCHEDULE_GPIPE, True), (pw.SCHEDULE_PER_MICROBATCH, False)):
        one = run_chain_gpu(pw, w, 2, M, pw.DISPATCH_OPBYOP, schedule, recompute, flags=pw.FLAG_WHOLE_LAYER)
        for dispatch in (pw.DISPATCH_ASYNC, pw.DISPATCH_GRAPH):
            lanes = run_chain_gpu(pw, w, 2, M, dispatch, schedule, recompute, flags=pw.FLAG_WHOLE_LAYER)
            for a, b in zip(one[0] + one[1], lanes[0] + lanes[1]):
                assert torch.isfinite(a.float()).all() and torch.equal(a, b)
            for l in range(2):
                assert all(torch.equal(a, b) for a, b in zip(one[2][l], lanes[2][l]))
