"""GeLU and its derivative far out, and the tanh form's distance from 64 bits."""
import math

import pytest
import torch

from tests.test_gpu_gelu import M, N, mean_error

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


def exact(x, act):
    """GeLU and its derivative in 64 bits."""
    if act == 0:
        cdf, pdf = 0.5 * torch.erfc(-x * 0.5 ** 0.5), torch.exp(-0.5 * x * x) / math.sqrt(2 * math.pi)
        return x * cdf, cdf + x * pdf
    z = math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)
    s = torch.sigmoid(2 * z)
    return x * s, s + x * s * torch.sigmoid(-2 * z) * 2 * math.sqrt(2 / math.pi) * (1 + 3 * 0.044715 * x * x)


def gelu(pw, A, B, act, n):
    u, a = (torch.empty((A.shape[0], n), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    bias = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
    pw.op_gemm(pw.GEMM_TN, pw.EPI_BIAS_GELU, A.shape[0], n, 8, A, 8, B, 8, u, n, bias=bias, aux_out=a, act=act)
    return u, a


def gelu_grad(pw, u, f, act):
    """f GeLU'(u), f of shape [rows, 1] + [1, columns]."""
    m, n = u.shape
    A, B = torch.zeros((m, 8), dtype=torch.bfloat16, device="cuda"), torch.zeros((8, n), dtype=torch.bfloat16, device="cuda")
    A[:, 0], A[:, 1], B[0], B[1] = f[0][:, 0], 1.0, 1.0, f[1][0]
    got = torch.empty((m, n), dtype=torch.bfloat16, device="cuda")
    pw.op_gemm(pw.GEMM_NN, pw.EPI_DGELU, m, n, 8, A, 8, B, n, got, n, aux_in=u, ld_aux=n, act=act)
    return got


def allowance(act, x, want, grad):
    """What the fp32 evaluation may be off by, before its rounding to bf16.  Body: a few roundings of 2^-24 and the fits' error, of |u| for GeLU
    and of 1 for the derivative.  Lower tail: the fits' error relative to the value (7.6e-5 for L; 1.7e-8, but at most 1 / x^2 of the value, for D; the
    tanh form has only roundings, 2^-24 of an exponent of up to 2^7), and beyond the fits, or where fp32 ends, no more than the value itself."""
    ax, aw = x.abs(), want.abs()
    body = (1.5e-7 if grad else 2e-7 * ax) + 0 * ax
    if act == 1:
        tail, end = 2e-5 * aw, 9.9
    elif grad:
        tail, end = torch.minimum(2e-8 + 0 * ax, aw / (x * x)), 9.5
    else:
        tail, end = 1.5e-4 * aw, 7.0
    return torch.where((x < -3), torch.where(ax <= end, tail, aw), body) + 1e-35


@pytest.mark.parametrize("act", [0, 1])
def test_every_exponent(pw, act):
    """All bf16 values from 2^-20 to the largest, both signs: bf16 of the exact value to half a spacing and what the evaluation may be off by, and the
    limits far out: u and 0 for GeLU, 1 and 0 for the derivative."""
    bits = torch.arange((127 - 20) << 7, 0x7f80, dtype=torch.int32, device="cuda")
    v = torch.cat([bits, bits + 0x8000]).to(torch.int16).view(torch.bfloat16)
    v = torch.cat([v, torch.zeros(-len(v) % 128, dtype=torch.bfloat16, device="cuda")])
    A, B = torch.zeros((len(v), 8), dtype=torch.bfloat16, device="cuda"), torch.zeros((128, 8), dtype=torch.bfloat16, device="cuda")
    A[:, 0], B[:, 0] = v, 1.0
    u, a = gelu(pw, A, B, act, 128)
    assert torch.equal(u[:, 77], v)
    one = torch.ones((len(v), 1), dtype=torch.bfloat16, device="cuda"), torch.zeros((1, 128), dtype=torch.bfloat16, device="cuda")
    d = gelu_grad(pw, u, one, act)
    x = v.double()
    far = x.abs() > 40
    for got, want, limit, grad in ((a, exact(x, act)[0], torch.where(x > 0, x, 0.0), False), (d, exact(x, act)[1], (x > 0).double(), True)):
        assert torch.equal(got[:, 0], got[:, 127])
        g = got[:, 5].double()
        assert ((g - limit).abs()[far] <= 1e-30 * limit.abs()[far] + 1e-30).all()
        near = ~far
        err, spacing = (g - want).abs(), torch.exp2(torch.floor(torch.log2(want.abs().clamp_min(2.0 ** -126))) - 7)
        bad = (err > 0.51 * spacing + allowance(act, x, want, grad)) & near
        assert not bad.any(), (x[bad][:8].tolist(), g[bad][:8].tolist(), want[bad][:8].tolist())


# a tile of its own, and CTA pairs
@pytest.mark.parametrize("m,n", [(128, 128), (4096, 4096)])
@pytest.mark.parametrize("act", [0, 1])
def test_infinities(pw, act, m, n):
    """What u times the distribution function gives: infinity at infinity, no number at minus infinity and for none."""
    A, B = torch.zeros((m, 8), dtype=torch.bfloat16, device="cuda"), torch.zeros((n, 8), dtype=torch.bfloat16, device="cuda")
    A[:, 0], B[:, 0] = 1.0, 1.0
    A[5, 0], A[70, 0], A[99, 0] = math.inf, -math.inf, math.nan
    u, a = gelu(pw, A, B, act, n)
    assert (u[5] == math.inf).all() and (u[70] == -math.inf).all() and torch.isnan(u[99]).all()
    assert (a[5] == math.inf).all() and torch.isnan(a[70]).all() and torch.isnan(a[99]).all()
    rest = torch.ones(m, dtype=torch.bool, device="cuda")
    rest[[5, 70, 99]] = False
    assert (a[rest] == torch.nn.functional.gelu(torch.ones((), device="cuda"), approximate="tanh" if act else "none").to(torch.bfloat16)).all()


# 1 - 2 / (exp(2 z) + 1) gives 3.4e-8 and 5.2e-8 root mean square before rounding, what is in use 1.8e-8 and 2.5e-8.  The mean of the
# magnitudes, which is measured here, is lower: 2.5e-9 and 2.0e-8 for what is in use.
def test_tanh_form(pw):
    g = torch.Generator(device="cuda").manual_seed(3)
    ri = lambda n, top: torch.randint(-top, top + 1, (n,), generator=g, device="cuda").double()
    A, B = (torch.zeros((n, 8), dtype=torch.bfloat16, device="cuda") for n in (M, N))
    A[:, 0], A[:, 1], A[:, 2] = ri(M, 255) * 2.0 ** -6, 1.0, ri(M, 31)          # exact sums whose low bits are spread
    B[:, 0], B[:, 1], B[:, 2] = 1.0, ri(N, 255) * 2.0 ** -14, ri(N, 31) * 2.0 ** -21
    err = mean_error(gelu(pw, A, B, 1, N)[1], exact(A.double() @ B.double().T, 1)[0])
    assert err < 3e-8, err
    f = torch.randint(128, 256, (M, 1), generator=g, device="cuda").double()
    e = torch.randint(0, 256, (1, N), generator=g, device="cuda").double() * 2.0 ** -8
    u = torch.randn((M, N), generator=g, device="cuda").to(torch.bfloat16)
    err = mean_error(gelu_grad(pw, u, (f, e), 1), (f + e) * exact(u.double(), 1)[1], 256.0) / f.mean().item()
    assert err < 4e-8, err
