"""The GEMM kernels of a layer request their weights before the kernel in front of them is complete: weights that were written just
before a call must still be the ones it uses."""
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


# every kind of GEMM kernel: K slices in a cluster, one tile a CTA, CTA pairs; the recomputing backward starts with a forward, the lean one makes its
# operands again on a second stream, one whose dx lies over dy starts with a weight gradient, and without CTA pairs all weight gradients are kernels of their own
@pytest.mark.parametrize("d,F,S,B,save,over,pair", [(256, 1024, 128, 2, "full", False, 1), (512, 2048, 256, 4, "recompute", False, 1), (1024, 4096, 512, 2, "full", False, 1),
                                                    (1024, 4096, 1024, 4, "recompute", False, 1), (256, 1024, 128, 2, "lean", False, 1), (1024, 4096, 1024, 2, "lean", True, 1),
                                                    (1024, 4096, 512, 2, "full", True, 1), (1024, 4096, 1024, 4, "full", False, 0), (512, 2048, 256, 4, "lean", True, 0)])
def test_weights_written_just_before(pw, d, F, S, B, save, over, pair):
    g = torch.Generator(device="cuda").manual_seed(d + S)
    T = S * B
    n = lambda *s: torch.randn(s, generator=g, device="cuda")
    shapes = ((d,), (d,), (3 * d, d), (3 * d,), (d, d), (d,), (d,), (d,), (F, d), (F,), (d, F), (d,))
    params = [(0.02 * n(*s)).to(torch.bfloat16) for s in shapes]
    start = [p.float() for p in params]
    layer = pw.Layer(d, d // 64, 64, F, S, B, flags=pw.FLAG_LEAN_CTX if save == "lean" else 0)
    x, dy0 = n(T, d).to(torch.bfloat16), n(T, d).to(torch.bfloat16)
    y, dy = torch.empty_like(x), dy0.clone()
    dx = dy if over else torch.empty_like(x)
    grads = [torch.zeros(s, device="cuda") for s in shapes]
    ctx = None if save == "recompute" else torch.empty(layer.ctx_bytes, dtype=torch.uint8, device="cuda")
    scratch = torch.empty(layer.scratch_bytes, dtype=torch.uint8, device="cuda")
    masters = [t.clone() for t in start]
    items = list(zip(params, masters, grads))
    fwd = lambda: layer.fwd(params, x, y, ctx, scratch)

    def bwd():
        if over:
            dy.copy_(dy0)
        layer.bwd(params, x, dy, dx, grads, False, ctx, scratch)

    # weights written in front of a forward and of a backward, and (last) behind a round
    parts = (fwd, bwd, lambda: pw.sgd_apply(items, 1e-4), fwd, lambda: pw.sgd_apply(items, 5e-5), bwd)

    def passes(how):
        out = []
        for p, m, t in zip(params, masters, start):
            m.copy_(t)
            p.copy_(t)
        torch.cuda.synchronize()
        graph = None
        if how == "replayed":
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                for part in parts:
                    part()
        for _ in range(6):
            if graph is not None:
                graph.replay()
            else:
                for part in parts:
                    part()
                    if how == "one by one":
                        torch.cuda.synchronize()
            out += [y.clone(), dx.clone()] + [t.clone() for t in grads]
            pw.sgd_apply(items, 2e-5)
            if how == "one by one":
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out

    pw.set_tuning(pw.TUNE_GEMM_PAIR, pair)
    try:
        want = passes("one by one")
        assert all(t.isfinite().all() for t in want) and not torch.equal(want[0], want[-len(want) // 6])
        for how in ("on", "on", "on", "replayed"):
            assert all(torch.equal(a, b) for a, b in zip(want, passes(how)))
    finally:
        pw.set_tuning(pw.TUNE_GEMM_PAIR, 1)
    assert layer.status() == (0, 0)


def test_language_model_step_with_weights_just_applied(pw):
    """The step's own kernels in front of the first layer (embedding) and behind the last (final LayerNorm, tied projection), with all weights written
    by the gradient apply just before."""
    L, V, d, F, S, B = 2, 512, 256, 1024, 128, 2
    g = torch.Generator(device="cuda").manual_seed(9)
    n = lambda *s: torch.randn(s, generator=g, device="cuda")
    shapes = ((d,), (d,), (3 * d, d), (3 * d,), (d, d), (d,), (d,), (d,), (F, d), (F,), (d, F), (d,))
    params = [[(0.02 * n(*s)).to(torch.bfloat16) for s in shapes] for _ in range(L)]
    ends = [(0.02 * n(V, d)).to(torch.bfloat16), (1 + 0.1 * n(d)).to(torch.bfloat16), (0.1 * n(d)).to(torch.bfloat16)]
    weights = [t for p in params for t in p] + ends
    start = [t.float() for t in weights]
    masters = [t.clone() for t in start]
    grads = [[torch.zeros(s, device="cuda") for s in shapes] for _ in range(L)]
    end_grads = [torch.zeros(t.shape, device="cuda") for t in ends]
    gradients = [t for p in grads for t in p] + end_grads
    ids, labels = (torch.randint(0, V, (B, S), generator=g, device="cuda", dtype=torch.int32) for _ in range(2))
    loss = torch.zeros(1, device="cuda")
    stage = pw.Stage(L, d, d // 64, 64, F, S, B)
    ws = torch.empty(stage.lm_workspace_bytes(V, False), dtype=torch.uint8, device="cuda")

    def steps(wait):
        out = []
        for w, m, t in zip(weights, masters, start):
            m.copy_(t)
            w.copy_(t)
        for _ in range(8):
            stage.lm_step(params, grads, ends, end_grads, ids, labels, loss, V, ws, False)
            if wait:
                torch.cuda.synchronize()
            pw.sgd_apply(list(zip(weights, masters, gradients)), 0.05)
            if wait:
                torch.cuda.synchronize()
            out += [loss.clone()] + [t.clone() for t in gradients]
        torch.cuda.synchronize()
        return out + [t.clone() for t in weights]

    want = steps(True)
    assert all(t.isfinite().all() for t in want) and want[0] > want[7 * (len(want) - len(weights)) // 8]
    for _ in range(3):
        assert all(torch.equal(a, b) for a, b in zip(want, steps(False)))
    assert stage.status() == (0, 0)
