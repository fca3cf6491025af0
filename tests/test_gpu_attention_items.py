"""Attention forward on both sides of the launcher's choice between pairs of query tiles and single ones (148 SMs)."""
import numpy as np
import pytest
import torch

from tests.gpu_util import ACT_TOL, ELEM_ACT, bf16_randn, elem_check, guard_alloc, np64, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("B,S,H,dh", [
    (1, 128, 3, 64),                              # one tile: pairs, whose second slot is idle
    (1, 256, 1, 128), (2, 384, 3, 64),            # singles of one, two and three key tiles
    (2, 1024, 16, 64), (3, 896, 9, 128),          # singles, more than one to a CTA: Q buffers, rings and counters go round
    (4, 640, 20, 64), (8, 512, 16, 128)])         # pairs, the last one incomplete; several to a CTA
def test_attention_fwd_items(pw, oracle64, B, S, H, dh):
    g = torch.Generator().manual_seed(S + H)
    d = H * dh
    qkv = bf16_randn((B * S, 3 * d), g)
    qkv[:, :2 * d] *= 3                           # the two slots' maxima differ by more than a rescale
    o, check_o = guard_alloc((B * S, d), torch.bfloat16)
    lse, check_l = guard_alloc((B, H, S), torch.float32)
    q = qkv.cuda()
    for _ in range(2):                            # the second launch finds the counters that the first one cleared
        o.zero_()
        pw.op_attention_fwd(q, B, S, H, dh, o, lse)
    torch.cuda.synchronize()
    assert pw.op_status() == (0, 0)
    check_o(); check_l()
    ow, lw = oracle64.attn_fwd(np64(qkv), B, S, H, dh)
    assert rel_l2(o, ow) < ACT_TOL
    elem_check(o, ow, "o", **ELEM_ACT)
    # scores are sums of dh products of exact bf16 values, good to dh * 2^-24 of sum |q k|, below 2^-13 here; 1e-3 as elsewhere
    assert np.abs(lse.double().cpu().numpy() - lw).max() < 1e-3
