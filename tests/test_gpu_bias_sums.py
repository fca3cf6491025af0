"""The two bias gradients of a layer that are column sums taken beside its weight gradients."""
import pytest
import torch

from paper_2203_12533_b200 import inputs
from tests.gpu_util import make_layer, run_layer_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


# one and several column blocks with a ragged last one; a few rows per warp, eight in flight with a remainder, one warp per block
@pytest.mark.parametrize("d,H,F,S,B", [(256, 4, 128, 128, 1), (256, 4, 384, 128, 1), (512, 4, 1920, 640, 3), (1024, 16, 4096, 1152, 3),
                                       (4096, 32, 16384, 256, 1)])
def test_column_sums(pw, d, H, F, S, B):
    w = inputs.Workload("sums", d, H, d // H, F, S, B)
    T = w.tokens
    params = [p.cuda() for p in inputs.layer_params(w, 0, 0, random_ln=True)]
    x, dy = (t.cuda().view(T, -1) for t in inputs.microbatch(w, 0, 0))
    layer = make_layer(pw, w)
    out = run_layer_gpu(pw, layer, params, x, dy)
    du = torch.empty((T, F), dtype=torch.bfloat16, device="cuda")
    u = layer.ctx_view(out["ctx"], "u")
    pw.op_gemm(pw.GEMM_NN, pw.EPI_DGELU, T, F, d, dy, d, params[pw.PARAM_NAMES.index("w_fc2")], F, du, F, aux_in=u, ld_aux=F)
    torch.cuda.synchronize()
    g = dict(zip(pw.PARAM_NAMES, out["grads"]))
    # fp32 sums in chains of at most T / 32 + 32 terms and a reduction: 2^-24 a step, on the sum of magnitudes
    err = (g["b_fc1"].double() - du.double().sum(0)).abs()
    assert (err <= (T / 32 + 64) * 2.0 ** -24 * du.double().abs().sum(0) + 1e-30).all()
    # the values' part is the column sum of dout over all queries, for every softmax row sums to one; bf16 P and dV: 2^-8 a term
    db = g["b_qkv"].double()
    assert torch.isfinite(db).all()
    p = dict(zip(pw.PARAM_NAMES, params))
    dout_sum = (g["b_o"].double() @ p["w_o"].double())
    rel = (db[2 * d:] - dout_sum).norm() / dout_sum.norm()
    assert rel < 0.02, rel
