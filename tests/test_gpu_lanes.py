"""A chain whose micro-batches take turns on several streams gives the bits of the chain on one stream.

OPBYOP runs on the calling stream alone; ASYNC and GRAPH use the lanes.  Micro-batch counts below, at and beyond the lane
count, and not a multiple of it."""
import pytest
import torch

from paper_2203_12533_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pw():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2203_12533_b200 import binding
    binding.lib()
    return binding


def streams_of(pw, call):
    """How many streams a chain call says that it uses."""
    lines = []
    pw.set_log(pw.LOG_INFO, lambda level, msg: lines.append(msg))
    try:
        call()
    finally:
        pw.set_log(pw.LOG_OFF)
    chains = [line for line in lines if line.startswith("pw_stage_run_chain:")]
    assert len(chains) == 1, lines
    return int(chains[0].split(", ")[-1].split()[0])


@pytest.mark.parametrize("width,heads,seq,batch,layers,M,flags", [
    (256, 4, 128, 2, 3, 1, 0), (256, 4, 128, 2, 3, 2, 0), (256, 4, 128, 1, 2, 5, 0), (256, 4, 128, 2, 3, 9, 0),     # four lanes
    (256, 4, 128, 2, 2, 6, "lean"), (256, 4, 128, 2, 3, 6, "whole"), (512, 8, 256, 2, 2, 3, "whole"),
    (1024, 8, 1024, 2, 2, 3, 0), (1024, 16, 1152, 1, 2, 2, 0)])                                                  # two lanes
@pytest.mark.parametrize("gpipe,recompute", [(True, True), (True, False), (False, True), (False, False)])
def test_lanes_change_no_bit(pw, width, heads, seq, batch, layers, M, flags, gpipe, recompute):
    w = inputs.Workload("lanes", width, heads, width // heads, 2 * width, seq, batch)
    flags = {"lean": pw.FLAG_LEAN_CTX, "whole": pw.FLAG_WHOLE_LAYER, 0: 0}[flags]
    schedule = pw.SCHEDULE_GPIPE if gpipe else pw.SCHEDULE_PER_MICROBATCH
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l, random_ln=True)] for l in range(layers)]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(M)])
    stage = pw.Stage(layers, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch, flags=flags)
    ws = torch.empty(stage.workspace_bytes(M, schedule, recompute), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()

    def chain(dispatch):
        ws.fill_(255)                                        # stale activations would not go unseen (bf16 NaN)
        ys, dxs = [torch.full_like(x, 7.0) for x in xs], [torch.full_like(x, 7.0) for x in xs]
        grads = [[torch.full(p.shape, 7.0, device="cuda") for p in ps] for ps in params]
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            n = streams_of(pw, lambda: stage.run_chain(params, grads, xs, dys, ys, dxs, ws, dispatch, schedule, recompute, stream=stream))
        assert n == (1 if dispatch == pw.DISPATCH_OPBYOP else min(M, 4 if w.tokens * width <= 256 * 256 else 2))
        torch.cuda.synchronize()
        assert stage.status() == (0, 0)
        return ys + dxs + [g for gs in grads for g in gs]

    ref = chain(pw.DISPATCH_OPBYOP)
    assert all(torch.isfinite(t).all() for t in ref)
    n0 = stage.launch_count()
    for dispatch in (pw.DISPATCH_ASYNC, pw.DISPATCH_GRAPH, pw.DISPATCH_ASYNC):
        for a, b in zip(ref, chain(dispatch)):
            assert torch.equal(a, b)
    assert stage.launch_count() == 4 * n0                    # every lane's launches are counted, a graph's too


def test_one_buffer_for_every_output_keeps_the_last_micro_batch(pw):
    """Overlapping buffers keep the chain on one stream: the last micro-batch's y is what stays."""
    w = inputs.Workload("lanes", 256, 4, 64, 512, 128, 2)
    M, L = 5, 2
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l)] for l in range(L)]
    grads = [[torch.zeros(p.shape, device="cuda") for p in ps] for ps in params]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(M)])
    stage = pw.Stage(L, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch)
    ws = torch.empty(stage.workspace_bytes(M, pw.SCHEDULE_GPIPE, True), dtype=torch.uint8, device="cuda")
    ys, dxs = [torch.empty_like(x) for x in xs], [torch.empty_like(x) for x in xs]
    chain = lambda ys: streams_of(pw, lambda: stage.run_chain(params, grads, xs, dys, ys, dxs, ws, pw.DISPATCH_ASYNC))
    assert chain(ys) == 4
    stage.set_side_stream(False)
    assert chain(ys) == 1
    stage.set_side_stream(True)
    y = torch.empty_like(xs[0])
    buf = torch.empty((w.tokens + 8, 256), dtype=torch.bfloat16, device="cuda")
    assert chain([y] * M) == 1
    part = [buf[:w.tokens]] + ys[1:-1] + [buf[8:]]           # the first and the last overlap by all but eight rows
    want = ys[-1].clone()
    assert chain(part) == 1
    torch.cuda.synchronize()
    assert torch.equal(y, want) and torch.equal(buf[8:], want)


@pytest.mark.parametrize("flags", ["", "whole"])
@pytest.mark.parametrize("dispatch", ["ASYNC", "GRAPH"])
def test_first_chain_of_a_stage_beside_a_busy_default_stream(pw, dispatch, flags):
    """The first chain call finds its lanes made: it allocates nothing, makes no handle and waits for nothing that the default
    stream still holds."""
    w = inputs.Workload("lanes", 256, 4, 64, 512, 128, 2)
    M, L = 6, 3
    flags = pw.FLAG_WHOLE_LAYER if flags else 0
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l, random_ln=True)] for l in range(L)]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(M)])

    def buffers():
        return ([torch.full_like(x, 7.0) for x in xs], [torch.full_like(x, 7.0) for x in xs],
                [[torch.full(p.shape, 7.0, device="cuda") for p in ps] for ps in params])

    def stage():
        return pw.Stage(L, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch, flags=flags)

    first = stage()
    ws = torch.empty(first.workspace_bytes(M, pw.SCHEDULE_GPIPE, True), dtype=torch.uint8, device="cuda")
    ys, dxs, grads = buffers()
    first.run_chain(params, grads, xs, dys, ys, dxs, ws, pw.DISPATCH_OPBYOP)
    ref = ys + dxs + [g for gs in grads for g in gs]
    ys, dxs, grads = buffers()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(1_500_000_000)                         # most of a second of work on the default stream
    done = torch.cuda.Event()
    done.record()
    st = stage()
    lines = []
    pw.set_log(pw.LOG_INFO, lambda level, msg: lines.append(msg))
    try:
        free = torch.cuda.mem_get_info()[0]
        st.run_chain(params, grads, xs, dys, ys, dxs, ws, getattr(pw, "DISPATCH_" + dispatch), stream=stream)
        if dispatch == "ASYNC":                              # (an instantiated graph is memory of its own)
            assert torch.cuda.mem_get_info()[0] == free
    finally:
        pw.set_log(pw.LOG_OFF)
    stream.synchronize()
    # all of it while the default stream was busy (a cooperative launch may wait for what that holds)
    assert flags == pw.FLAG_WHOLE_LAYER or not done.query()
    assert lines and not any("_create" in line for line in lines), lines
    for a, b in zip(ref, ys + dxs + [g for gs in grads for g in gs]):
        assert torch.equal(a, b)
    assert st.status() == (0, 0)


def test_whole_layer_launches_share_the_sms_by_the_lanes_in_use(pw):
    """One stage, chains of one to six micro-batches in turn: each number of lanes has grids of its own size, whose barrier words must not mix."""
    w = inputs.Workload("lanes", 256, 4, 64, 512, 128, 2)
    L = 2
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l, random_ln=True)] for l in range(L)]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(6)])
    stage = pw.Stage(L, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch, flags=pw.FLAG_WHOLE_LAYER)
    ws = torch.empty(stage.workspace_bytes(6), dtype=torch.uint8, device="cuda")
    for M in (2, 4, 3, 1, 2, 6, 3):
        out = []
        for dispatch in (pw.DISPATCH_OPBYOP, pw.DISPATCH_ASYNC):
            ys, dxs = [torch.empty_like(x) for x in xs[:M]], [torch.empty_like(x) for x in xs[:M]]
            grads = [[torch.empty(p.shape, device="cuda") for p in ps] for ps in params]
            n = streams_of(pw, lambda: stage.run_chain(params, grads, xs[:M], dys[:M], ys, dxs, ws, dispatch))
            assert n == (1 if dispatch == pw.DISPATCH_OPBYOP else min(M, 4))
            torch.cuda.synchronize()
            assert stage.status() == (0, 0)
            out.append(ys + dxs + [g for gs in grads for g in gs])
        for a, b in zip(*out):
            assert torch.equal(a, b), M


@pytest.mark.parametrize("gpipe,recompute", [(True, True), (False, False)])
def test_a_workspace_for_fewer_streams_is_enough(pw, gpipe, recompute):
    """From one stream's size on every workspace is taken, nothing is written behind it, and no bit changes."""
    w = inputs.Workload("lanes", 256, 4, 64, 512, 128, 2)
    M, L = 6, 3
    schedule = pw.SCHEDULE_GPIPE if gpipe else pw.SCHEDULE_PER_MICROBATCH
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l, random_ln=True)] for l in range(L)]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(M)])
    stage = pw.Stage(L, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch)
    full = stage.workspace_bytes(M, schedule, recompute)
    stage.set_side_stream(False)
    one = stage.workspace_bytes(M, schedule, recompute)
    stage.set_side_stream(True)
    assert one < full == stage.workspace_bytes(M, schedule, recompute)
    ws = torch.empty(full + 1024, dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    ref = None
    for dispatch, nbytes in [(pw.DISPATCH_OPBYOP, one), (pw.DISPATCH_ASYNC, full)] + [
            (d, n) for n in (one, one + (full - one) // 3 - 1, one + (full - one) // 3, one + (full - one) // 3 * 2, full - 1)
            for d in (pw.DISPATCH_ASYNC, pw.DISPATCH_GRAPH)]:
        ws.fill_(255)
        ys, dxs = [torch.empty_like(x) for x in xs], [torch.empty_like(x) for x in xs]
        grads = [[torch.empty(p.shape, device="cuda") for p in ps] for ps in params]
        torch.cuda.synchronize()
        n = streams_of(pw, lambda: stage.run_chain(params, grads, xs, dys, ys, dxs, ws, dispatch, schedule, recompute, stream=stream,
                                                   workspace_bytes=nbytes))
        assert n == (1 if dispatch == pw.DISPATCH_OPBYOP else 1 + (nbytes - one) * 3 // (full - one))
        torch.cuda.synchronize()
        assert stage.status() == (0, 0) and (ws[nbytes:] == 255).all()
        out = ys + dxs + [g for gs in grads for g in gs]
        ref = out if ref is None else ref
        for a, b in zip(ref, out):
            assert torch.equal(a, b)
    for dispatch in (pw.DISPATCH_OPBYOP, pw.DISPATCH_ASYNC):
        with pytest.raises(pw.PwError) as e:
            stage.run_chain(params, grads, xs, dys, ys, dxs, ws, dispatch, schedule, recompute, workspace_bytes=one - 1)
        assert e.value.status == 3


@pytest.mark.parametrize("tied", ["layers", "one_vector", "partly"])
def test_layers_that_share_gradient_buffers_keep_their_order(pw, tied):
    """Two layers that write one gradient buffer: who writes when decides what stays, so the chain keeps to one stream."""
    w = inputs.Workload("lanes", 256, 4, 64, 512, 128, 2)
    M, L = 6, 4
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l, random_ln=True)] for l in range(L)]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(M)])
    stage = pw.Stage(L, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch)
    ws = torch.empty(stage.workspace_bytes(M), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.Stream()
    ref = None
    for dispatch in [pw.DISPATCH_OPBYOP] + [pw.DISPATCH_ASYNC, pw.DISPATCH_GRAPH] * 3:
        ys, dxs = [torch.empty_like(x) for x in xs], [torch.empty_like(x) for x in xs]
        grads = [[torch.empty(p.shape, device="cuda") for p in ps] for ps in params]
        if tied == "layers":
            grads[2] = grads[0]
        elif tied == "one_vector":
            grads[3][3] = grads[1][3]                        # b_qkv
        else:
            both = torch.empty(w.d_model + 64, device="cuda")
            grads[0][0], grads[1][7] = both[:w.d_model], both[64:]           # ln1_gamma of one over ln2_beta of the other
        torch.cuda.synchronize()
        assert streams_of(pw, lambda: stage.run_chain(params, grads, xs, dys, ys, dxs, ws, dispatch, stream=stream)) == 1
        torch.cuda.synchronize()
        assert stage.status() == (0, 0)
        out = ys + dxs + [g for gs in grads for g in gs]
        ref = out if ref is None else ref
        for a, b in zip(ref, out):
            assert torch.equal(a, b)


def test_a_chain_first_called_inside_a_capture_uses_its_lanes(pw):
    w = inputs.Workload("lanes", 256, 4, 64, 512, 128, 2)
    M, L = 5, 2
    params = [[p.cuda() for p in inputs.layer_params(w, 0, l, random_ln=True)] for l in range(L)]
    xs, dys = zip(*[[t.cuda().view(w.tokens, -1) for t in inputs.microbatch(w, 0, m)] for m in range(M)])
    out = []
    for captured in (False, True):
        stage = pw.Stage(L, w.d_model, w.n_heads, w.head_dim, w.d_ff, w.seq_len, w.batch)
        ws = torch.empty(stage.workspace_bytes(M), dtype=torch.uint8, device="cuda")
        ys, dxs = [torch.full_like(x, 7.0) for x in xs], [torch.full_like(x, 7.0) for x in xs]
        grads = [[torch.full(p.shape, 7.0, device="cuda") for p in ps] for ps in params]
        torch.cuda.synchronize()
        call = lambda: stage.run_chain(params, grads, xs, dys, ys, dxs, ws, pw.DISPATCH_ASYNC)
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                assert streams_of(pw, call) == 4
            graph.replay()
        else:
            call()
        torch.cuda.synchronize()
        assert stage.status() == (0, 0)
        out.append(ys + dxs + [g for gs in grads for g in gs])
    for a, b in zip(*out):
        assert torch.equal(a, b)
