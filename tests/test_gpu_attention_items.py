"""Attention forward and backward with few and many work items; forward on both sides of the launcher's choice between pairs of query tiles and single ones (148 SMs)."""
import numpy as np
import pytest
import torch

from tests.gpu_util import ACT_TOL, ELEM_ACT, GRAD_TOL, bf16_randn, elem_check, guard_alloc, np64, rel_l2

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
    (4, 640, 20, 64), (8, 512, 16, 128),          # pairs, the last one incomplete; several to a CTA
    (8, 640, 13, 128)])                           # the same with two score buffers: a tile alone in its item, and tile B's last one
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


@pytest.mark.parametrize("B,S,H,dh", [
    (1, 128, 2, 64),                              # one query tile, no second one
    (4, 640, 20, 64), (5, 640, 10, 128),          # several items to a CTA, the first of them with a single query tile
    (3, 768, 17, 64)])                            # and with pairs only: buffers and rings of three and five go round
def test_attention_bwd_items(pw, oracle64, B, S, H, dh):
    g = torch.Generator().manual_seed(S + H + 1)
    d = H * dh
    qkv, dout = bf16_randn((B * S, 3 * d), g), bf16_randn((B * S, d), g)
    q, do = qkv.cuda(), dout.cuda()
    o = torch.empty((B * S, d), dtype=torch.bfloat16, device="cuda")
    lse = torch.empty((B, H, S), device="cuda")
    delta = torch.empty((B, H, S), device="cuda")
    pw.op_attention_fwd(q, B, S, H, dh, o, lse)
    got = []
    for _ in range(2):
        dqkv, check = guard_alloc((B * S, 3 * d), torch.bfloat16)
        pw.op_attention_bwd(q, o, do, lse, B, S, H, dh, dqkv, delta)
        torch.cuda.synchronize()
        assert pw.op_status() == (0, 0)
        check()
        got.append(dqkv)
    assert torch.equal(got[0], got[1])
    dw = oracle64.attn_bwd(np64(qkv), np64(dout), B, S, H, dh)
    for name, sl in (("dq", slice(0, d)), ("dk", slice(d, 2 * d)), ("dv", slice(2 * d, 3 * d))):
        assert rel_l2(got[0][:, sl], dw[:, sl]) < GRAD_TOL, name
        # The errors are bf16 roundings of P, dS and the result, relative and independent, so every 128 x dh tile keeps the
        # bound of the whole up to the scatter of its 2^13 or more errors; a wrong tile is off by about 1.  (A bound for single
        # elements fits the 5e4 of the small tests; the worst of these 3e6 lies a few percent further out in the tail.)
        diff = (got[0][:, sl].double().cpu().numpy() - dw[:, sl]).reshape(B * S // 128, 128, H, dh)
        want = np.asarray(dw[:, sl]).reshape(diff.shape)
        tile = np.sqrt((diff ** 2).sum((1, 3)) / (want ** 2).sum((1, 3)))
        assert tile.max() < 2 * GRAD_TOL, (name, tile.max())


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("B,S,H,dh", [(1, 128, 2, 64), (2, 384, 3, 128), (3, 640, 17, 64)])
def test_attention_bwd_takes_any_float_pointers(pw, B, S, H, dh, shift):
    """lse and delta at any multiple of four bytes give the bits of 16-byte aligned ones."""
    g = torch.Generator().manual_seed(S + shift)
    d, n = H * dh, B * H * S
    q, do = bf16_randn((B * S, 3 * d), g).cuda(), bf16_randn((B * S, d), g).cuda()
    o = torch.empty((B * S, d), dtype=torch.bfloat16, device="cuda")
    got = []
    for at in [(0, 0), (shift, 0), (0, shift), (shift, (shift + 1) % 4)]:
        lse, delta = (torch.full((n + 4,), float("nan"), device="cuda")[k:k + n].view(B, H, S) for k in at)
        dqkv, check = guard_alloc((B * S, 3 * d), torch.bfloat16)
        pw.op_attention_fwd(q, B, S, H, dh, o, lse)
        pw.op_attention_bwd(q, o, do, lse, B, S, H, dh, dqkv, delta)
        torch.cuda.synchronize()
        assert pw.op_status() == (0, 0)
        check()
        got.append(dqkv)
    assert torch.isfinite(got[0]).all()
    for t in got[1:]:
        assert torch.equal(t, got[0])


@pytest.mark.parametrize("B,S,H,dh", [(2, 4096, 16, 64), (2, 1024, 16, 64), (4, 1024, 16, 64), (1, 2048, 16, 128)])
def test_attention_same_bits_every_time(pw, B, S, H, dh):
    """Thousands of launches back to back: warps of a tile that drift apart must not change a bit."""
    g = torch.Generator(device="cuda").manual_seed(S + dh)
    d = H * dh
    qkv, dout = (torch.randn((B * S, n), generator=g, device="cuda").to(torch.bfloat16) for n in (3 * d, d))
    n_out = 8
    outs = [(torch.empty((B * S, d), dtype=torch.bfloat16, device="cuda"), torch.empty((B, H, S), device="cuda")) for _ in range(n_out)]
    ref = None
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(250):
        for o, lse in outs:                       # nothing between them: the next launch's warps are already on the SMs
            pw.op_attention_fwd(qkv, B, S, H, dh, o, lse)
        if ref is None:
            ref = [t.clone() for t in outs[0]]
        for o, lse in outs:
            wrong += (o != ref[0]).sum() + (lse != ref[1]).sum()
    o, lse = ref
    ref = None
    for _ in range(50):
        dqkv, delta = torch.empty_like(qkv), torch.empty_like(lse)
        pw.op_attention_bwd(qkv, o, dout, lse, B, S, H, dh, dqkv, delta)
        ref = dqkv if ref is None else ref
        wrong += (dqkv != ref).sum()
    torch.cuda.synchronize()
    assert pw.op_status() == (0, 0)
    assert wrong.item() == 0


@pytest.mark.parametrize("B,S,H", [(8, 1024, 16), (16, 640, 16), (9, 384, 33)])
def test_attention_fwd_same_bits_128_wide_pairs(pw, B, S, H):
    """Pairs of query tiles, even and odd numbers of key tiles.  The two threads of a row swap their maxima through one set of
    words, so neither may write its next maximum before the other has read the last one: on every key tile of an item without a
    tile B, and in front of tile B's diagonal one, the scores that it comes from may already be there.  Scores as large as these make the maximum jump by more than a rescale."""
    g = torch.Generator(device="cuda").manual_seed(S)
    d = H * 128
    qkv = torch.randn((B * S, 3 * d), generator=g, device="cuda").to(torch.bfloat16)
    qkv[:, :2 * d] *= 3
    outs = [(torch.empty((B * S, d), dtype=torch.bfloat16, device="cuda"), torch.empty((B, H, S), device="cuda")) for _ in range(4)]
    ref = None
    wrong = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(250):
        for o, lse in outs:
            pw.op_attention_fwd(qkv, B, S, H, 128, o, lse)
        if ref is None:
            ref = [t.clone() for t in outs[0]]
        for o, lse in outs:
            wrong += (o != ref[0]).sum() + (lse != ref[1]).sum()
    torch.cuda.synchronize()
    assert pw.op_status() == (0, 0)
    assert wrong.item() == 0
