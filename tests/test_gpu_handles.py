"""A handle is ready when its create call returns, on whatever stream its first call runs.

Its counters are zeroed by then: a kernel on a non-blocking stream waits for nothing that the default stream still holds."""
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


def busy_default_stream():
    """Most of a second of work on the default stream, and an event behind it."""
    torch.cuda.synchronize()
    torch.cuda._sleep(1_500_000_000)
    done = torch.cuda.Event()
    done.record()
    return done


@pytest.mark.parametrize("flags", ["", "lean", "whole"])
def test_first_call_of_a_layer_beside_a_busy_default_stream(pw, flags):
    w = inputs.Workload("ready", 256, 4, 64, 1024, 256, 2)
    flags = {"": 0, "lean": pw.FLAG_LEAN_CTX, "whole": pw.FLAG_WHOLE_LAYER}[flags]
    params = [p.cuda() for p in inputs.layer_params(w, 0, 0, random_ln=True)]
    x, dy = (t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, 0))
    first = make_layer(pw, w, flags=flags)
    ref = run_layer_gpu(pw, first, params, x, dy)
    y, dx = torch.empty_like(x), torch.empty_like(x)
    grads = [torch.full_like(g, float("nan")) for g in ref["grads"]]
    ctx, scratch = torch.empty_like(ref["ctx"]), torch.empty_like(ref["scratch"])
    stream = torch.cuda.Stream()
    done = busy_default_stream()
    layer = make_layer(pw, w, flags=flags)
    layer.fwd(params, x, y, ctx, scratch, stream=stream)
    layer.bwd(params, x, dy, dx, grads, False, ctx, scratch, stream=stream)
    stream.synchronize()
    # all of it while the default stream was busy (a cooperative launch may wait for what that holds)
    assert flags == pw.FLAG_WHOLE_LAYER or not done.query()
    assert torch.equal(y.cpu(), ref["y"].cpu()) and torch.equal(dx.cpu(), ref["dx"].cpu())
    for name, a, b in zip(pw.PARAM_NAMES, grads, ref["grads"]):
        assert torch.equal(a, b), name
    assert layer.status() == (0, 0)
