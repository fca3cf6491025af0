"""GEMMs with few output tiles: one cluster per tile, the K range cut into slices inside it.

The sizes sit at the edges of the launcher's choices (148 SMs): a single tile, every number of K slices with and
without a ragged last block of 64, tile counts of exactly one per SM and one more, ragged M and N."""
import pytest
import torch

from tests.gpu_util import guard_alloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


SIZES = [(8, 8, 8), (128, 64, 64), (264, 256, 768), (200, 328, 1544), (1024, 512, 1600), (392, 136, 776),
         (512, 2368, 1024),      # 148 tiles of 128 x 64
         (512, 2432, 1032),      # four more than one per SM, ragged K
         (1024, 1152, 2056),     # 72 tiles of 128 x 128, cut in two
         (512, 4736, 520),       # 148 tiles of 128 x 128
         (1016, 4728, 1096),     # two per SM, ragged edges
         (1024, 4864, 512),      # more than two per SM: the persistent kernel
         (1016, 3072, 1096), (1920, 3464, 1288)]     # its 192-wide tiles: one round, a ragged second one


@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("kind", ["bias", "resid", "gelu", "dgrad", "dgelu", "rowdot", "wgrad"])
def test_few_tiles(pw, M, N, K, kind):
    if kind == "rowdot" and (N % 64 or M % 8):
        pytest.skip("heads are 64 wide")
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    ri = lambda *s: torch.randint(-2, 3, s, generator=g, device="cuda").to(torch.bfloat16)
    nt, nn = kind == "wgrad", kind in ("dgrad", "dgelu", "rowdot")
    A, B = (ri(K, M) if nt else ri(M, K)), (ri(K, N) if nt or nn else ri(N, K))
    bias, aux = ri(N), ri(M, N)
    want = (A.double().T if nt else A.double()) @ (B.double() if nt or nn else B.double().T)
    C, check = guard_alloc((M, N), torch.float32 if nt else torch.bfloat16)
    out2, check2 = guard_alloc((M, N), torch.bfloat16)
    lda, ldb = (M if nt else K), (N if nt or nn else K)

    def run():
        if kind == "rowdot":
            rd = torch.empty((1, N // 64, M), device="cuda")
            pw.op_gemm_rowdot(M, N, K, A, K, B, N, C, N, aux, N, 64, M, rd)
            return rd
        layout = pw.GEMM_NT if nt else pw.GEMM_NN if nn else pw.GEMM_TN
        epi = {"bias": pw.EPI_BIAS, "resid": pw.EPI_BIAS_RESID, "gelu": pw.EPI_BIAS_GELU, "dgrad": pw.EPI_NONE,
               "dgelu": pw.EPI_DGELU, "wgrad": pw.EPI_F32}[kind]
        pw.op_gemm(layout, epi, M, N, K, A, lda, B, ldb, C, N, bias=bias, aux_in=aux, ld_aux=N,
                   aux_out=out2 if kind == "gelu" else None)
        return None

    rd = run()
    torch.cuda.synchronize()
    assert pw.op_status() == (0, 0)
    check(); check2()
    # small integers: products and sums are exact in fp32, so the result is exact up to the bf16 store
    if kind in ("bias", "resid", "gelu"):
        want = want + bias.double() + (aux.double() if kind == "resid" else 0)
    if kind == "dgelu":
        u = aux.double().requires_grad_()
        torch.nn.functional.gelu(u).sum().backward()
        want = want * u.grad
        # one bf16 rounding (2^-9) of a product with a derivative good to 1e-6
        assert ((C.double() - want).abs() <= 2.0 ** -8 * want.abs() + 1e-5 * want.abs().max()).all()
    else:
        assert torch.equal(C.double(), want if nt else want.to(torch.bfloat16).double())
    if kind == "gelu":
        a = torch.nn.functional.gelu(want)
        assert ((out2.double() - a).abs() <= 2.0 ** -8 * a.abs() + 1e-5).all()
    if kind == "rowdot":
        dots = (want * aux.double()).view(M, N // 64, 64).sum(-1).T
        assert torch.equal(rd[0].double(), dots.float().double())
    if nt:                                                   # accumulate adds, twice the sum is exact too
        pw.op_gemm(pw.GEMM_NT, pw.EPI_F32, M, N, K, A, M, B, N, C, N, accumulate=True)
        torch.cuda.synchronize()
        assert torch.equal(C.double(), 2 * want)
    elif kind != "rowdot":                                   # the same bits again
        first = C.clone()
        run()
        torch.cuda.synchronize()
        assert torch.equal(C, first)


@pytest.mark.parametrize("knob,value", [("TUNE_GEMM_BN", 128), ("TUNE_GEMM_BN", 192), ("TUNE_GEMM_BN", 256), ("TUNE_GEMM_PAIR", 0)])
@pytest.mark.parametrize("kind", ["bias", "resid", "gelu", "dgrad", "dgelu", "rowdot", "wgrad"])
@pytest.mark.parametrize("M,N,K", [(200, 5056, 264), (1000, 5184, 2056)])     # less than one pair's rows; tiles cut in two, ragged K
def test_tile_widths(pw, M, N, K, kind, knob, value):
    before = pw.get_tuning(getattr(pw, knob))
    pw.set_tuning(getattr(pw, knob), value)
    pw.set_tuning(pw.TUNE_GEMM_SPLIT_MIN_K, 8)
    try:
        test_few_tiles(pw, M, N, K, kind)
    finally:
        pw.set_tuning(getattr(pw, knob), before)
        pw.set_tuning(pw.TUNE_GEMM_SPLIT_MIN_K, 64)
