"""LayerNorm on both sides of the launchers' choices: backward with eight rows a CTA or persistent CTAs, forward with few CTAs or many."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


# one row, a full and a started eighth, every width of the eight-row form, and the last and first token counts around its bounds
@pytest.mark.parametrize("T,d", [(1, 256), (8, 512), (9, 768), (63, 1024), (1025, 1280), (40, 1536), (17, 1792), (129, 2048), (128, 2048),
                                 (2048, 256), (2049, 256), (4096, 768), (4097, 768), (2048, 2048), (2049, 2048)])
@pytest.mark.parametrize("sums", [True, False])
def test_against_64_bits(pw, T, d, sums):
    g = torch.Generator(device="cuda").manual_seed(T + d)
    n = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    x, dh, resid, gamma = n(T, d), n(T, d), n(T, d), n(d)
    mu, rstd = x.double().mean(1).float(), (x.double().var(1, unbiased=False) + 1e-5).rsqrt().float()
    pad = 64
    buf = torch.full((T + 2, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    dx = buf[1:-1]
    out = [torch.full((d + 2 * pad,), 3.0, device="cuda") for _ in range(4)]
    vec = [t[pad:-pad] for t in out]
    part = torch.empty(pw.op_layernorm_bwd_scratch_bytes(T, d), dtype=torch.uint8, device="cuda")
    for accumulate in (False, True):
        pw.op_layernorm_bwd(dh, x, mu, rstd, gamma, resid, dx, *(vec if sums else vec[:2] + [None, None]), accumulate, part)
    torch.cuda.synchronize()
    X, D, R = x.double(), dh.double(), resid.double()
    xhat, gg = (X - mu.double()[:, None]) * rstd.double()[:, None], D * gamma.double()
    want = R + rstd.double()[:, None] * (gg - gg.mean(1, keepdim=True) - xhat * (gg * xhat).mean(1, keepdim=True))
    # half a spacing of bf16 and fp32 rounding of row sums of d terms
    assert ((dx.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-4).all()
    assert torch.isnan(buf[0].float()).all() and torch.isnan(buf[-1].float()).all()
    terms = [D * xhat, D] + ([R, dx.double()] if sums else [])
    for v, o, t in zip(vec, out, terms):
        # twice the sum (overwritten, then added to): chains of at most T terms in fp32, each rounding 2^-24 of the magnitudes so far
        assert ((v.double() - 2 * t.sum(0)).abs() <= 2 * (T + 64) * 2.0 ** -24 * t.abs().sum(0) + 1e-6).all()
        assert (o[:pad] == 3.0).all() and (o[-pad:] == 3.0).all()


# every number of 16-byte pieces a lane, one and several warps a row; the last token count with no more CTAs than SMs and the first with more
@pytest.mark.parametrize("T,d", [(1, 256), (9, 512), (77, 768), (1184, 1024), (1185, 1024), (300, 1280), (64, 1536), (33, 1792), (1184, 2048), (1185, 2048),
                                 (592, 4096), (593, 4096), (5, 5120), (148, 8192), (149, 8192)])
def test_forward_against_64_bits(pw, T, d):
    g = torch.Generator(device="cuda").manual_seed(T * 3 + d)
    n = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    x, gamma, beta = n(T, d), n(d), n(d)
    buf = torch.full((T + 2, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    h, mu, rstd = buf[1:-1], torch.empty(T, device="cuda"), torch.empty(T, device="cuda")
    pw.op_layernorm_fwd(x, gamma, beta, 1e-5, h, mu, rstd)
    torch.cuda.synchronize()
    X = x.double()
    m, r = X.mean(1), (X.var(1, unbiased=False) + 1e-5).rsqrt()
    want = (X - m[:, None]) * r[:, None] * gamma.double() + beta.double()
    # half a spacing of bf16, and fp32 rounding of sums of d terms
    assert ((h.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-5).all()
    assert (mu.double() - m).abs().max() < 1e-6 and ((rstd.double() - r) / r).abs().max() < 1e-6
    assert torch.isnan(buf[0].float()).all() and torch.isnan(buf[-1].float()).all()


# one row of eight, a started eighth, and the persistent form
@pytest.mark.parametrize("T,d", [(1, 256), (9, 512), (17, 1280), (3, 4096)])
def test_infinite_gamma(pw, T, d):
    """An infinity in gamma takes whole rows of dx to infinities (and to no numbers): their column sums are those of the rows that are there."""
    g = torch.Generator(device="cuda").manual_seed(T * 5 + d)
    n = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    row, gamma = n(1, d), n(d)
    x, dh, resid = (t.expand(T, d).contiguous() for t in (row, n(1, d), n(1, d)))
    gamma[7] = float("inf")
    mu, rstd = x.double().mean(1).float(), (x.double().var(1, unbiased=False) + 1e-5).rsqrt().float()
    dx = torch.empty_like(x)
    vec = [torch.zeros(d, device="cuda") for _ in range(4)]
    part = torch.empty(pw.op_layernorm_bwd_scratch_bytes(T, d), dtype=torch.uint8, device="cuda")
    pw.op_layernorm_bwd(dh, x, mu, rstd, gamma, resid, dx, *vec, False, part)
    torch.cuda.synchronize()
    want = dx.float().sum(0)
    assert torch.isinf(want).sum() > d // 8                    # (equal rows: no infinities of both signs in a column)
    assert torch.equal(torch.isnan(vec[3]), torch.isnan(want)) and torch.equal(vec[3][torch.isinf(want)], want[torch.isinf(want)])
    assert all(torch.isfinite(v).all() for v in vec[:3])
