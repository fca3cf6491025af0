"""Timed cases: what programs built on this library have it do, through its public entry points.

A case is a dict of plain values:

  kind      "layer"    one training call of a decoder layer: Layer.fwd, then Layer.bwd
            "forward"  Layer.fwd alone, nothing saved for a backward (evaluation, scoring)
            "chain"    a pipeline stage: Stage.run_chain over its micro-batches
            "lm"       a training step of a language model: Stage.lm_step, then sgd_apply
  width, head_dim, ff, seq, batch     d_model, width of a head, d_ff, sequence length, sequences per call
  act       "erf" or "tanh" GeLU
  save      what the backward finds from the forward: "full", "lean" or "recompute" (chain and lm: only the layers' inputs)
  whole     one kernel launch per layer call (FLAG_WHOLE_LAYER: small shapes with 64-wide heads)
  layers, micro_batches, dispatch, schedule      chain (lm: layers alone)
  vocab     lm

Widths are those of the workloads in ``paper_2203_12533_b200/inputs.py`` and of the tests, or others
that the library takes (d_model in multiples of 256, above 2048 of 512 and above 4096 of 1024; d_ff
and the sequence length in multiples of 128).
"""
from __future__ import annotations

import torch

from paper_2203_12533_b200 import binding as pw

_ACT = {"erf": pw.ACT_GELU_ERF, "tanh": pw.ACT_GELU_TANH}
_DISPATCH = {"opbyop": pw.DISPATCH_OPBYOP, "async": pw.DISPATCH_ASYNC, "graph": pw.DISPATCH_GRAPH}
_SCHEDULE = {"gpipe": pw.SCHEDULE_GPIPE, "per_microbatch": pw.SCHEDULE_PER_MICROBATCH}
_LEARNING_RATE = 0.01
_DEVICE = "cuda"
_graph_stream = None


def _layer(name, width, head_dim, ff, seq, batch, act="erf", save="full", whole=False):
    return {"name": name, "kind": "layer", "width": width, "head_dim": head_dim, "ff": ff, "seq": seq, "batch": batch,
            "act": act, "save": save, "whole": whole}


def _forward(name, width, head_dim, ff, seq, batch, act="erf"):
    return {"name": name, "kind": "forward", "width": width, "head_dim": head_dim, "ff": ff, "seq": seq, "batch": batch,
            "act": act, "save": "full", "whole": False}


def _chain(name, layers, micro_batches, width, head_dim, ff, seq, batch, act="erf", save="recompute", whole=False,
           dispatch="async", schedule="gpipe"):
    return {"name": name, "kind": "chain", "layers": layers, "micro_batches": micro_batches, "width": width,
            "head_dim": head_dim, "ff": ff, "seq": seq, "batch": batch, "act": act, "save": save, "whole": whole,
            "dispatch": dispatch, "schedule": schedule}


def _lm(name, layers, vocab, width, head_dim, ff, seq, batch, act="erf", save="full"):
    return {"name": name, "kind": "lm", "layers": layers, "vocab": vocab, "width": width, "head_dim": head_dim, "ff": ff,
            "seq": seq, "batch": batch, "act": act, "save": save, "whole": False}


def listed():
    return [
        # The smallest call: 256 tokens through the 256-wide layer, forward and backward, called one by one.
        # Launches and their latency are all there is.
        _layer("layer_w256_t256", 256, 64, 1024, 128, 2),
        # Chained small computations as one program: 8 layers x 8 micro-batches at that width, one launch per
        # layer call, the whole chain replayed as a graph.
        _chain("chain_small_whole_graph", 8, 8, 256, 64, 1024, 128, 2, whole=True, dispatch="graph"),
        # A small model's layer on a small micro-batch (1024 tokens): too few output tiles to fill the chip.
        _layer("layer_w1024_t1024", 1024, 64, 4096, 512, 2),
        # Odd sizes: a width, a hidden size, a sequence length and a batch that divide into nothing evenly.
        _layer("layer_w1280_odd", 1280, 128, 3456, 640, 3, act="tanh"),
        # Scoring one long prompt with the 2048-wide layer (forward only, nothing kept).
        _forward("forward_w2048_s2048", 2048, 128, 8192, 2048, 1),
        # The ordinary call: the 2048-wide layer of the three-billion-parameter decoder, 8 sequences of 1024.
        _layer("layer_w2048_t8192", 2048, 128, 8192, 1024, 8),
        # Long context with 64-wide heads: attention weighs as much as the matrix products; lean save set.
        _layer("layer_long_context_lean", 1024, 64, 4096, 4096, 2, save="lean"),
        # The widest layer on one sequence: large weights, few tokens.
        _layer("layer_w8192_t2048", 8192, 128, 32768, 2048, 1),
        # A stage of a mid-sized model that keeps its activations, one micro-batch at a time.
        _chain("chain_w1024_saved", 4, 4, 1024, 64, 4096, 1024, 2, save="full", schedule="per_microbatch"),
        # The largest: a four-layer stage at width 4096, activations recomputed, GPipe order, two of its micro-batches.
        _chain("chain_w4096_recompute", 4, 2, 4096, 128, 16384, 2048, 4),
        # A small language model's whole training step, gradients applied.
        _lm("lm_small", 6, 8192, 512, 64, 2048, 256, 4),
        # The 12-layer language model's whole training step, gradients applied.
        _lm("lm_w1024_v32768", 12, 32768, 1024, 64, 4096, 1024, 16),
    ]


def draw(rng):
    """One more case of the same ranges; never dearer than the dearest listed one."""
    most = max(_executed_flops(c) for c in listed())
    while True:
        kind = rng.choice(("layer", "layer", "layer", "forward", "chain", "lm"))
        width = 2 ** rng.uniform(8, 13 if kind in ("layer", "forward") else 12)
        step = 256 if width <= 2048 else 512 if width <= 4096 else 1024
        width = step * round(width / step)
        ff = 128 * max(2, round(width * rng.uniform(2.0, 4.5) / 128))
        seq = 128 * round(2 ** rng.uniform(0, 5))
        batch = max(1, round(2 ** rng.uniform(8, 14.5) / seq))
        head_dim, act = rng.choice((64, 128)), rng.choice(("erf", "erf", "tanh"))
        if kind == "forward":
            c = _forward("", width, head_dim, ff, seq, batch, act)
        elif kind == "layer":
            c = _layer("", width, head_dim, ff, seq, batch, act, rng.choice(("full", "full", "lean", "recompute")))
        elif kind == "chain":
            c = _chain("", rng.randint(2, 8), rng.randint(1, 8), width, head_dim, ff, seq, batch, act,
                       rng.choice(("full", "lean", "recompute")), False, rng.choice(("opbyop", "async", "graph")),
                       rng.choice(("gpipe", "per_microbatch")))
        else:
            c = _lm("", rng.randint(2, 12), 8 * round(2 ** rng.uniform(7, 12)), width, head_dim, ff, seq, batch, act,
                    rng.choice(("full", "full", "lean", "recompute")))
        del c["name"]
        small = width <= 512 and head_dim == 64 and seq <= 1024 and (seq * batch // 64) * (width // 64) <= 1024
        if kind in ("layer", "chain") and small and c["save"] != "lean":
            c["whole"] = rng.random() < 0.5
        # Several layers' passes are long enough as they are: leave out what would fill the card with saved activations.
        saved = c.get("layers", 1) * c.get("micro_batches", 1) * 2 * seq * batch * (7 * width + 2 * ff)
        if _executed_flops(c) <= most and saved <= 24e9:
            return c


# ---------------------------------------------------------------------------------------------------- work
def _tokens(c):
    return c["seq"] * c["batch"]


def _param_count(c):
    d, f = c["width"], c["ff"]
    return 4 * d * d + 2 * d * f + 9 * d + f


def _forward_flops(c):
    """One layer on one micro-batch; attention at the visible pairs (token i sees i + 1 keys)."""
    t, d = _tokens(c), c["width"]
    return 8.0 * t * d * d + 4.0 * t * d * c["ff"] + 2.0 * t * (c["seq"] + 1) * d


def _model_flops(c):
    """Forward and backward without anything done twice."""
    f = _forward_flops(c)
    if c["kind"] == "forward":
        return f
    return 3.0 * f + _tokens(c) * (c["seq"] + 1.0) * c["width"]          # attention's backward: five products for the forward's two


def _head_flops(c):
    return 6.0 * _tokens(c) * c["width"] * c["vocab"] if c["kind"] == "lm" else 0.0


def _executed_flops(c):
    again = _forward_flops(c) if c["save"] == "recompute" and c["kind"] != "forward" else 0.0
    return c.get("layers", 1) * c.get("micro_batches", 1) * (_model_flops(c) + again) + _head_flops(c)


def work(case):
    """What one pass cannot do without: every input read once, every result written once, no recomputation."""
    c = case
    layers, micro = c.get("layers", 1), c.get("micro_batches", 1)
    rows = 2.0 * _tokens(c) * c["width"]                                 # one activation tensor, bf16
    params = layers * _param_count(c)
    flops = layers * micro * _model_flops(c) + _head_flops(c)
    if c["kind"] == "forward":
        return {"bytes": 2.0 * params + 2 * rows, "flops": flops}
    if c["kind"] != "lm":
        return {"bytes": 6.0 * params + 4 * micro * rows, "flops": flops}     # weights in, fp32 gradients out; x, dy, y, dx
    params += c["vocab"] * c["width"] + 2 * c["width"]
    return {"bytes": 16.0 * params + 8.0 * _tokens(c), "flops": flops}   # + the fp32 master in and out, new bf16 weights out


def tolerance(case):
    """bf16 operands, bf16 activations handed from step to step, fp32 sums.  Against the same layers in fp64 the worst
    output of one layer is off by 3e-3 to 6e-3 (largest element 0.06 of the rms), of a stack of layers by 7e-3 to 1e-2
    (0.29): about four times that for one layer, twice to three times for a stack."""
    return {"rel": 2e-2, "max": 0.25} if case.get("layers", 1) == 1 else {"rel": 3e-2, "max": 0.6}


# ---------------------------------------------------------------------------------------------------- state
def _param_shapes(c):
    d, f = c["width"], c["ff"]
    return ((d,), (d,), (3 * d, d), (3 * d,), (d, d), (d,), (d,), (d,), (f, d), (f,), (d, f), (d,))


def _draw_params(c, layers, gen):
    """The twelve tensors of a layer for all layers, stacked along a first dimension."""
    sigma = 0.01 if c["width"] >= 8192 else 0.02
    out = []
    for name, shape in zip(pw.PARAM_NAMES, _param_shapes(c)):
        t = torch.empty((layers, *shape), dtype=torch.bfloat16, device=_DEVICE)
        for l in range(layers):
            v = torch.randn(shape, generator=gen, device=_DEVICE)
            t[l] = 1.0 + 0.1 * v if "gamma" in name else 0.1 * v if "beta" in name else sigma * v
        out.append(t)
    return out


def _normal(shape, gen):
    return torch.randn(shape, generator=gen, device=_DEVICE).to(torch.bfloat16)


def _bytes(n):
    return torch.empty(n, dtype=torch.uint8, device=_DEVICE)


def _flags(c):
    return (pw.FLAG_LEAN_CTX if c["save"] == "lean" else 0) | (pw.FLAG_WHOLE_LAYER if c["whole"] else 0)


def _per_layer(stacked):
    """The stacked tensors as the library takes them: twelve for each layer."""
    return [[t[l] for t in stacked] for l in range(stacked[0].shape[0])]


def prepare(case, seed):
    global _graph_stream
    c = case
    gen = torch.Generator(device=_DEVICE)
    gen.manual_seed(seed)
    layers = c.get("layers", 1)
    shape = (c["width"], c["width"] // c["head_dim"], c["head_dim"], c["ff"], c["seq"], c["batch"])
    s = {"case": c, "params": _draw_params(c, layers, gen)}
    s["layer_params"] = _per_layer(s["params"])
    if c["kind"] != "forward":
        s["grads"] = [torch.zeros(p.shape, dtype=torch.float32, device=_DEVICE) for p in s["params"]]
        s["layer_grads"] = _per_layer(s["grads"])
    if c["kind"] in ("layer", "forward"):
        s["layer"] = pw.Layer(*shape, act=_ACT[c["act"]], flags=_flags(c))
        s["scratch"] = _bytes(s["layer"].scratch_bytes)
        s["x"] = _normal((_tokens(c), c["width"]), gen)
        s["y"] = torch.empty_like(s["x"])
        if c["kind"] == "layer":
            s["ctx"] = _bytes(s["layer"].ctx_bytes) if c["save"] != "recompute" else None
            s["dy"] = _normal((_tokens(c), c["width"]), gen)
            s["dx"] = torch.empty_like(s["x"])
        return s
    s["stage"] = pw.Stage(layers, *shape, act=_ACT[c["act"]], flags=_flags(c))
    recompute = c["save"] == "recompute"
    if c["kind"] == "chain":
        m, schedule = c["micro_batches"], _SCHEDULE[c["schedule"]]
        s["xs"] = [_normal((_tokens(c), c["width"]), gen) for _ in range(m)]
        s["dys"] = [_normal((_tokens(c), c["width"]), gen) for _ in range(m)]
        s["ys"], s["dxs"] = [torch.empty_like(t) for t in s["xs"]], [torch.empty_like(t) for t in s["xs"]]
        s["workspace"] = _bytes(s["stage"].workspace_bytes(m, schedule, recompute))
        s["stream"] = None
        if c["dispatch"] == "graph":                                     # a graph cannot be captured on the default stream
            if _graph_stream is None:
                _graph_stream = torch.cuda.Stream()
            s["stream"] = _graph_stream
    else:
        v, d = c["vocab"], c["width"]
        s["ends"] = [0.02 * torch.randn((v, d), generator=gen, device=_DEVICE), 1.0 + 0.1 * torch.randn(d, generator=gen, device=_DEVICE),
                     0.1 * torch.randn(d, generator=gen, device=_DEVICE)]
        s["ends"] = [t.to(torch.bfloat16) for t in s["ends"]]
        s["end_grads"] = [torch.zeros(t.shape, dtype=torch.float32, device=_DEVICE) for t in s["ends"]]
        s["weights"], s["gradients"] = s["params"] + s["ends"], s["grads"] + s["end_grads"]
        s["masters"] = [t.float() for t in s["weights"]]
        s["ids"], s["labels"] = (torch.randint(0, v, (c["batch"], c["seq"]), generator=gen, device=_DEVICE, dtype=torch.int32) for _ in range(2))
        s["loss"] = torch.zeros(1, device=_DEVICE)
        s["workspace"] = _bytes(s["stage"].lm_workspace_bytes(v, recompute))
    return s


# ---------------------------------------------------------------------------------------------------- one pass
def run(state):
    s, c = state, state["case"]
    params = s["layer_params"]
    if c["kind"] == "forward":
        s["layer"].fwd(params[0], s["x"], s["y"], None, s["scratch"])
        return {"y": s["y"]}
    grads = s["layer_grads"]
    if c["kind"] == "layer":
        s["layer"].fwd(params[0], s["x"], s["y"], s["ctx"], s["scratch"])
        s["layer"].bwd(params[0], s["x"], s["dy"], s["dx"], grads[0], False, s["ctx"], s["scratch"])
        return {"y": s["y"], "dx": s["dx"], "grads": grads[0]}
    recompute = c["save"] == "recompute"
    if c["kind"] == "chain":
        s["stage"].run_chain(params, grads, s["xs"], s["dys"], s["ys"], s["dxs"], s["workspace"], _DISPATCH[c["dispatch"]],
                             _SCHEDULE[c["schedule"]], recompute, stream=s["stream"])
        return {"ys": s["ys"], "dxs": s["dxs"], "grads": s["grads"]}
    s["stage"].lm_step(params, grads, s["ends"], s["end_grads"], s["ids"], s["labels"], s["loss"], c["vocab"], s["workspace"], recompute)
    pw.sgd_apply(list(zip(s["weights"], s["masters"], s["gradients"])), _LEARNING_RATE)
    return {"loss": s["loss"], "grads": s["gradients"], "weights": s["weights"], "masters": s["masters"]}
