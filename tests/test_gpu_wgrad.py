"""Weight gradients: up to four products in one launch, as one pool of 256-row tiles.

Integer operands make every sum exact.  The sizes take each tile width, fewer tiles than the 74 CTA pairs, exactly one
round, a remainder, and ragged M, N and K; the layers give pools of four products (three where dx overwrites dy)."""
import pytest
import torch

from paper_2203_12533_b200 import inputs
from tests.gpu_util import guard_alloc, make_layer, run_layer_gpu, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("M,N,K", [(2048, 2048, 1024), (1800, 2056, 1032), (2304, 1536, 4104), (2560, 2304, 2056), (4736, 1024, 520),
                                   (3840, 3464, 3080), (4872, 4608, 1544), (264, 4096, 8200)])
def test_products_are_exact(pw, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, B = (torch.randint(-2, 3, (K, n), generator=g, device="cuda").to(torch.bfloat16) for n in (M, N))
    want = A.double().T @ B.double()
    for accumulate in (False, True):
        C, check = guard_alloc((M, N), torch.float32)
        C.fill_(3.0)
        for _ in range(2 if accumulate else 1):
            pw.op_gemm(pw.GEMM_NT, pw.EPI_F32, M, N, K, A, M, B, N, C, N, accumulate=accumulate)
        torch.cuda.synchronize()
        assert pw.op_status() == (0, 0)
        check()
        assert torch.equal(C.double(), 2 * want + 3 if accumulate else want)


@pytest.mark.parametrize("alias", [False, True], ids=["dx", "dx_over_dy"])
@pytest.mark.parametrize("d,H,F,S,B", [(256, 4, 512, 128, 1), (512, 4, 2048, 256, 4), (1280, 10, 3456, 640, 3), (768, 12, 1920, 1152, 1)])
@pytest.mark.parametrize("lean", [False, True], ids=["full", "lean"])
def test_pool_of_a_layer(pw, d, H, F, S, B, alias, lean):
    """dW2 = dy^T a from the saved activation (fp64), and every gradient equal to the same layer's without aliasing."""
    w = inputs.Workload("pool", d, H, d // H, F, S, B)
    params = [p.cuda() for p in inputs.layer_params(w, 0, 0, random_ln=True)]
    x, dy = (t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, 0))
    layer = make_layer(pw, w, flags=pw.FLAG_LEAN_CTX if lean else 0)
    ref = run_layer_gpu(pw, layer, params, x, dy)
    y, ctx = torch.empty_like(x), torch.empty(layer.ctx_bytes, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(layer.scratch_bytes, dtype=torch.uint8, device="cuda")
    grads = [torch.full_like(g, float("nan")) for g in ref["grads"]]
    g = dy.clone()
    dx = g if alias else torch.empty_like(x)
    layer.fwd(params, x, y, ctx, scratch)
    a = torch.nn.functional.gelu(layer.ctx_view(ctx, "u").double()).to(torch.bfloat16) if lean else layer.ctx_view(ctx, "a")
    layer.bwd(params, x, g, dx, grads, False, ctx, scratch)
    torch.cuda.synchronize()
    assert layer.status() == (0, 0) and torch.equal(dx, ref["dx"])
    for name, g0, g1 in zip(pw.PARAM_NAMES, ref["grads"], grads):
        assert torch.equal(g0, g1), name
    # fp32 sums of T products of bf16 values; lean: a's bf16 roundings of two GeLU forms differ by a tie here and there
    assert rel_l2(grads[10], dy.double().T @ a.double()) < (1e-3 if lean else 1e-5)


@pytest.mark.parametrize("alias", [False, True], ids=["dx", "dx_over_dy"])
def test_pool_without_cta_pairs(pw, alias):
    """PW_TUNE_GEMM_PAIR = 0 reaches the weight gradients of a layer: four launches of single-CTA tiles, the same fp32 sums."""
    w = inputs.Workload("pool", 512, 4, 128, 2048, 256, 4)
    params = [p.cuda() for p in inputs.layer_params(w, 0, 0, random_ln=True)]
    x, dy = (t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, 0))
    layer = make_layer(pw, w)
    y, ctx = torch.empty_like(x), torch.empty(layer.ctx_bytes, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(layer.scratch_bytes, dtype=torch.uint8, device="cuda")
    launches = {}
    for value in (1, 0):
        grads = [torch.full(p.shape, float("nan"), device="cuda") for p in params]
        g = dy.clone()
        pw.set_tuning(pw.TUNE_GEMM_PAIR, value)
        try:
            layer.fwd(params, x, y, ctx, scratch)
            before = layer.launch_count()
            layer.bwd(params, x, g, g if alias else torch.empty_like(x), grads, False, ctx, scratch)
            launches[value] = layer.launch_count() - before
        finally:
            pw.set_tuning(pw.TUNE_GEMM_PAIR, 1)
        torch.cuda.synchronize()
        assert layer.status() == (0, 0) and all(torch.isfinite(t).all() for t in grads)
        # fp32 sums of T products of bf16 values, as above
        assert rel_l2(grads[10], dy.double().T @ layer.ctx_view(ctx, "a").double()) < 1e-5
    assert launches[0] == launches[1] + (2 if alias else 3)
