"""How far GeLU and its derivative are from 64 bits, seen through bf16 results.

A bf16 result differs from the rounded 64-bit value where that lies within the fp32 error of a rounding boundary, which has
probability error / spacing: the mean of (differs) x spacing over many values is the mean absolute error before rounding."""
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


# Hastings' five terms give 1.08e-7 and 5.4e-8 here with a correctly rounded reciprocal, 1.06e-7 and 5.7e-8 with one to an ulp, six fitted
# terms 2.5e-8 and 2.8e-8; the polynomials in the exponent that are in use 6.4e-9 and 1.8e-8, of which the roundings of the last products are most.
# The bounds lie between.
M, N = 4096, 16384


def mean_error(got, want, scale=1.0):
    """Estimate of the mean absolute error that `got` had before it was rounded to bf16."""
    right = want.to(torch.float32).to(torch.bfloat16)        # (64 -> 32 -> 16 bits: 2^-24 of a spacing's chance to round twice)
    spacing = torch.exp2(torch.floor(torch.log2(want.abs().clamp_min(2.0 ** -100))) - 7)
    # a few values beside a boundary, not wrong ones: no result is off by more than the one step
    assert ((got.double() - want).abs() <= 0.51 * spacing + scale * 1e-6).all()
    return ((got != right) * spacing).mean().item()


def test_gelu(pw):
    """GeLU of fp32 sums whose low bits are spread: a_m 2^-6 + b_n 2^-14 + c_m d_n 2^-21."""
    g = torch.Generator(device="cuda").manual_seed(1)
    ri = lambda n, top: torch.randint(-top, top + 1, (n,), generator=g, device="cuda").double()
    A, B = (torch.zeros((n, 8), dtype=torch.bfloat16, device="cuda") for n in (M, N))
    A[:, 0], A[:, 1], A[:, 2] = ri(M, 255) * 2.0 ** -6, 1.0, ri(M, 31)
    B[:, 0], B[:, 1], B[:, 2] = 1.0, ri(N, 255) * 2.0 ** -14, ri(N, 31) * 2.0 ** -21
    bias = torch.zeros(N, dtype=torch.bfloat16, device="cuda")
    u, got = (torch.empty((M, N), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    x = torch.empty((M, N), device="cuda")
    pw.op_gemm(pw.GEMM_NT, pw.EPI_F32, M, N, 8, A.T.contiguous(), M, B.T.contiguous(), N, x, N)
    assert torch.equal(x.double(), A.double() @ B.double().T)                # the sums are exact
    pw.op_gemm(pw.GEMM_TN, pw.EPI_BIAS_GELU, M, N, 8, A, 8, B, 8, u, N, bias=bias, aux_out=got)
    err = mean_error(got, torch.nn.functional.gelu(x.double()))
    assert err < 5e-8, err


def test_gelu_derivative(pw):
    """GeLU'(u) times f_m + e_n 2^-8 (128 <= f < 256): the product's own rounding is at most 2^-24 of it."""
    g = torch.Generator(device="cuda").manual_seed(2)
    f = torch.randint(128, 256, (M, 1), generator=g, device="cuda").double()
    e = torch.randint(0, 256, (1, N), generator=g, device="cuda").double() * 2.0 ** -8
    A, B = torch.zeros((M, 8), dtype=torch.bfloat16, device="cuda"), torch.zeros((8, N), dtype=torch.bfloat16, device="cuda")
    A[:, 0], A[:, 1], B[0], B[1] = f[:, 0], 1.0, 1.0, e[0]
    u = torch.randn((M, N), generator=g, device="cuda").to(torch.bfloat16)
    got = torch.empty((M, N), dtype=torch.bfloat16, device="cuda")
    pw.op_gemm(pw.GEMM_NN, pw.EPI_DGELU, M, N, 8, A, 8, B, N, got, N, aux_in=u, ld_aux=N)
    x = u.double()
    want = 0.5 * torch.erfc(-x * 0.5 ** 0.5) + x * torch.exp(-0.5 * x * x) * 0.3989422804014327
    err = mean_error(got, (f + e) * want, 256.0) / f.mean().item()
    assert err < 4e-8, err
