"""nf_block_step runs what a layer does behind its forward pass beside the next layers; nf_layer_step runs the auxiliary gradients beside
the rest.  Neither may change a bit against the same layers stepped one after the other, whatever the caller's buffers share."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = {
    "bf16": [(3, 64, 32, 32, False), (64, 64, 32, 32, False), (64, 128, 32, 16, True), (128, 128, 16, 16, False)],
    "f32": [(3, 8, 16, 4, False), (8, 8, 16, 4, False), (8, 8, 16, 8, True)],
    "same": [(64, 64, 16, 16, False)] * 5,
}


def _block(kind, N, seed, host_io=0):
    import torch
    from paper_2402_14139_b200 import nf
    nf.nf_set_stream(torch.cuda.current_stream())
    gen = torch.Generator(device="cuda").manual_seed(seed)
    layers = []
    for i, (Cin, Cout, S, F, pool) in enumerate(SHAPES[kind]):
        L = nf.Layer(Cin, Cout, S, S, F, 10, N, maxpool=pool, dtype=nf.NF_F32 if kind == "f32" else nf.NF_BF16, host_io=host_io if i == 0 else 0)
        for name, fan in (("W", 9 * Cin), ("Wa", 9 * Cout), ("Wf", 4 * F)):
            L.set_param(name, (torch.randn(L.shapes[name], generator=gen, device="cuda") * (2.0 / fan) ** 0.5).cpu().numpy())
        layers.append(L)
    Cin, _, S, _, _ = SHAPES[kind][0]
    x = torch.randn((N, S, S, Cin), generator=gen, device="cuda").to(layers[0].tdtype)
    y = torch.randint(0, 10, (N,), generator=gen, device="cuda", dtype=torch.int32)
    return nf, layers, nf.Block(layers), x, y


def _state(layers):
    return [L.get_param(k, kind) for L in layers for k in ("W", "gamma", "Wa", "ba", "Wf", "bf") for kind in (0, 0x200)] + \
        [L.get_param("rmean") for L in layers]


def _one_by_one(layers, x, y, loss, acts, steps):
    for _ in range(steps):
        cur = x
        for i, L in enumerate(layers):
            L.step(cur, y, 0.05, loss[i:i + 1], acts[i])
            cur = acts[i]


def _in_one_stream(nf, layers, x, y, loss, acts, steps):
    """The same with per-operation timing on, which keeps every launch of a step in the caller's stream."""
    nf.nf_trace_enable(True)
    try:
        _one_by_one(layers, x, y, loss, acts, steps)
    finally:
        nf.nf_trace_enable(False)


def _same(a, b):
    assert all((p == q).all() for p, q in zip(a, b))


@pytest.mark.parametrize("how", ["step", "graph", "other stream", "host", "layers"])
@pytest.mark.parametrize("kind,N", [("bf16", 96), ("bf16", 7), ("f32", 8), ("f32", 1535), ("f32", 1536), ("same", 40)])
def test_steps_have_the_bits_of_one_stream(kind, N, how):
    import torch
    nf, ref, _, x, y = _block(kind, N, 3)
    loss = torch.zeros(len(ref), device="cuda")
    acts = [L.new_act() for L in ref]
    _in_one_stream(nf, ref, x, y, loss, acts, 3)
    nf, layers, block, x, y = _block(kind, N, 3, 2 if how == "host" else 0)
    got, act = torch.zeros(len(ref), device="cuda"), layers[-1].new_act()
    if how == "graph":
        block.step(x, y, 0.05, got, act)
        g = block.capture(x, y, 0.05, got, act)
        for _ in range(2):
            g.replay()
    elif how == "layers":
        _one_by_one(layers, x, y, got, [L.new_act() for L in layers[:-1]] + [act], 3)
    elif how == "host":
        xh, yh, got = x.cpu().pin_memory(), y.cpu().pin_memory(), got.cpu().pin_memory()
        for _ in range(3):
            block.step_host_next(xh, yh, 0.05, got, xh, yh)
    else:
        s = torch.cuda.Stream() if how == "other stream" else torch.cuda.current_stream()
        s.wait_stream(torch.cuda.current_stream())
        nf.nf_set_stream(s)
        for _ in range(3):
            block.step(x, y, 0.05, got, act)
        torch.cuda.current_stream().wait_stream(s)
        nf.nf_set_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert torch.equal(got.cuda(), loss)
    assert how == "host" or torch.equal(act, acts[-1])
    _same(_state(layers), _state(ref))
    assert all(L.status() == 0 for L in layers)


def test_buffers_that_share_memory_keep_the_order_of_one_stream():
    """act_out in the input's place, and a shortcut that is a view of an earlier layer's buffer: single steps of the same calls agree."""
    import torch
    N = 40
    nf, ref, _, x, y = _block("same", N, 5)
    loss, acts = torch.zeros(len(ref), device="cuda"), [L.new_act() for L in ref]
    for c in range(2):
        ref[3].set_skip(ref[0].stored("dy") if c else None)
        xr = x.clone()
        cur = xr
        for i, L in enumerate(ref):
            out = xr if i == len(ref) - 1 else acts[i]
            L.step(cur, y, 0.05, loss[i:i + 1], out)
            cur = out
    nf, layers, block, x, y = _block("same", N, 5)
    got = torch.zeros(len(ref), device="cuda")
    for c in range(2):
        layers[3].set_skip(layers[0].stored("dy") if c else None)
        xb = x.clone()
        block.step(xb, y, 0.05, got, xb)
    torch.cuda.synchronize()
    assert torch.equal(xb, xr) and torch.equal(got, loss)
    _same(_state(layers), _state(ref))


def test_a_call_that_fails_half_way_leaves_the_stream_in_order():
    import torch
    nf, layers, block, x, y = _block("bf16", 16, 7)
    act = torch.empty(layers[-1].new_act().numel() + 8, dtype=torch.bfloat16, device="cuda")
    loss = torch.zeros(len(layers), device="cuda")
    with pytest.raises(nf.NfError):        # the last layer refuses its output's address; the ones before it have run
        block.step(x, y, 0.05, loss, act[1:])
    first = loss.clone()
    block.step(x, y, 0.05, loss, act)      # no update was made by the first call
    torch.cuda.synchronize()
    assert torch.equal(first[:-1], loss[:-1])


def test_lanes_of_many_layers_come_and_go():
    """More layers than streams are kept for; the ones that get a used stream step as the first ones did."""
    import torch
    nf, layers, block, x, y = _block("f32", 8, 9)
    loss = torch.zeros(len(layers), device="cuda")
    block.step(x, y, 0.05, loss)
    want = _state(layers)
    for _ in range(3):
        many = [_block("f32", 8, 9) for _ in range(12)]
        for _, ls, b, xx, yy in many:
            b.step(xx, yy, 0.05, torch.zeros(len(ls), device="cuda"))
        for _, ls, b, _, _ in many:
            _same(_state(ls), want)
            b.close()
            for L in ls:
                L.close()


def test_layers_that_go_while_a_capture_holds_their_lanes():
    """More layers than lanes are kept for, closed before the capture that has stepped them ends: the graph is whole, and its replay does
    what the same steps one after the other do."""
    import torch
    nf, ref, _, x, y = _block("f32", 8, 13)
    loss, act = torch.zeros(1, device="cuda"), ref[0].new_act()
    ref[0].step(x, y, 0.05, loss, act)
    many = [_block("f32", 8, 13)[1][0] for _ in range(40)]
    got, acts = torch.zeros(len(many), device="cuda"), [L.new_act() for L in many]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        nf.nf_set_stream(torch.cuda.current_stream())
        for i, L in enumerate(many):
            L.step(x, y, 0.05, got[i:i + 1], acts[i])
        grads = [L.dp_buffer(2) for L in many]
        for L in many:          # the handles only: their memory stays
            L.close()
    nf.nf_set_stream(torch.cuda.current_stream())
    g.replay()
    torch.cuda.synchronize()
    assert bool((got == loss).all()) and all(torch.equal(a, act) for a in acts)
    assert all(torch.equal(v, ref[0].dp_buffer(2)) for v in grads)
    _, fresh, block, x, y = _block("f32", 8, 13)    # and the lanes serve again
    block.step(x, y, 0.05, torch.zeros(len(fresh), device="cuda"))
    torch.cuda.synchronize()
    assert torch.equal(fresh[0].dp_buffer(2), ref[0].dp_buffer(2))


class _Recording:
    """A capture of one stream, which others may run beside."""

    def __init__(self, stream):
        from cuda.bindings import runtime as rt
        self.rt, self.stream = rt, stream
        self._do("cudaStreamBeginCapture", stream.cuda_stream, rt.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal)

    def _do(self, name, *args):
        err, *out = getattr(self.rt, name)(*args)
        assert err == self.rt.cudaError_t.cudaSuccess, (name, err)
        return out[0] if len(out) == 1 else out

    def end(self):
        self.graph = self._do("cudaStreamEndCapture", self.stream.cuda_stream)

    def replay(self):
        self._do("cudaGraphLaunch", self._do("cudaGraphInstantiate", self.graph, 0), self.stream.cuda_stream)

    def kernel_priorities(self):
        rt = self.rt
        nodes = self._do("cudaGraphGetNodes", self.graph, self._do("cudaGraphGetNodes", self.graph)[1])[0]
        kernels = [n for n in nodes if self._do("cudaGraphNodeGetType", n) == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel]
        assert len(kernels) >= 10 * len(SHAPES["bf16"])
        return {self._do("cudaGraphKernelNodeGetAttribute", n, rt.cudaLaunchAttributeID.cudaLaunchAttributePriority).priority for n in kernels}


@pytest.mark.parametrize("call", ["block", "layers"])
def test_an_ordinary_call_while_a_capture_holds_the_lanes(call):
    """Handles that a capture on one stream has stepped, stepped on another stream before it ends, and in a capture of a third one: what is
    recorded runs when its graph does, the ordinary step at once."""
    import torch
    nf, ref, _, x, y = _block("bf16", 24, 15)
    loss, acts = torch.zeros(len(ref), device="cuda"), [L.new_act() for L in ref]
    nf, layers, block, x, y = _block("bf16", 24, 15)
    got, out = torch.zeros(len(ref), device="cuda"), [L.new_act() for L in layers]

    def step(stream):
        nf.nf_set_stream(stream)
        if call == "block":
            block.step(x, y, 0.05, got, out[-1])
        else:
            _one_by_one(layers, x, y, got, out, 1)

    step(torch.cuda.current_stream())
    torch.cuda.synchronize()
    s1, s2, s3 = (torch.cuda.Stream() for _ in range(3))
    g = _Recording(s1)
    step(s1)
    step(s2)
    h = _Recording(s3)
    step(s3)
    step(s1)
    h.end()
    g.end()
    torch.cuda.synchronize()
    nf.nf_set_stream(torch.cuda.current_stream())
    _one_by_one(ref, x, y, loss, acts, 2)
    _same(_state(layers), _state(ref))
    for graph, steps in ((h, 1), (g, 2)):
        graph.replay()
        torch.cuda.synchronize()
        _one_by_one(ref, x, y, loss, acts, steps)
        _same(_state(layers), _state(ref))
    assert torch.equal(got, loss) and torch.equal(out[-1], acts[-1])
    assert all(L.status() == 0 for L in layers)


@pytest.mark.parametrize("call", ["block", "layers"])
def test_side_streams_have_the_priority_of_the_callers_stream(call):
    """Every kernel that a step records has the priority of the stream that it was called on, as a step in one stream does."""
    import torch
    nf, layers, block, x, y = _block("bf16", 24, 17)
    loss, acts = torch.zeros(len(layers), device="cuda"), [L.new_act() for L in layers]
    block.step(x, y, 0.05, loss)
    torch.cuda.synchronize()
    for prio in (0, -1, 0):
        s = torch.cuda.Stream(priority=prio)
        rec = _Recording(s)
        nf.nf_set_stream(s)
        if call == "block":
            block.step(x, y, 0.05, loss, acts[-1])
        else:
            _one_by_one(layers, x, y, loss, acts, 1)
        rec.end()
        nf.nf_set_stream(torch.cuda.current_stream())
        assert rec.kernel_priorities() == {prio}


@pytest.mark.parametrize("kind", ["bf16", "f32"])
@pytest.mark.parametrize("where", ["dy", "da", "dz"])
def test_activation_in_a_buffer_that_the_step_writes_later(kind, where):
    """act_out in the layer's own gradient buffers, or in the place of dz: the step reads it before it is written over."""
    import torch
    nf, ref, _, x, y = _block(kind, 24, 11)
    nf, layers, _, _, _ = _block(kind, 24, 11)
    loss, got = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    cur = x
    for R, L in zip(ref, layers):
        act = R.new_act()
        if where == "dz" and not L.maxpool:
            dz = L.new_act()
            L.set_skip_grad(dz)
            R.set_skip_grad(R.new_act())
            out = dz
        else:
            out = L.stored("dy" if where == "dz" else where).flatten()[:act.numel()]
        for _ in range(2):
            R.step(cur, y, 0.05, loss, act)
            L.step(cur, y, 0.05, got, out)
        assert torch.equal(loss, got)
        cur = act
    torch.cuda.synchronize()
    _same(_state(layers), _state(ref))


def _own_memory(L, name, bytes_on):
    """An activation-shaped view of the layer's workspace, `bytes_on` bytes into one of its tensors."""
    base = L.stored(name).data_ptr() - L.ws.data_ptr() + bytes_on
    n = L.N * L.Ha * L.Wa * L.Cout
    return L.ws[base:base + n * 2].view(L.tdtype).view(L.N, L.Ha, L.Wa, L.Cout)


@pytest.mark.parametrize("name,quarters", [("da", 0.125), ("da", 0.5), ("da", 0.875), ("dy", 0), ("dy", 0.5), ("dy", 1), ("dy", 1.5), ("dy", 2.75), ("dy", 3)])
def test_activation_of_a_pooled_layer_anywhere_in_its_own_gradients(name, quarters):
    """act_out at any place in da (and on into the activation buffer behind it) or in dy: the winners that the layer keeps for its backward
    pass lie elsewhere."""
    import torch
    nf, ref, _, _, y = _block("bf16", 24, 19)
    nf, layers, _, _, _ = _block("bf16", 24, 19)
    R, L = ref[2], layers[2]
    assert L.maxpool
    x = torch.randn((24, 32, 32, 64), generator=torch.Generator(device="cuda").manual_seed(19), device="cuda").clamp_min(0).bfloat16()
    loss, got, act = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda"), R.new_act()
    out = _own_memory(L, name, int(quarters * act.numel() * 2))
    for _ in range(2):
        R.step(x, y, 0.05, loss, act)
        L.step(x, y, 0.05, got, out)
    torch.cuda.synchronize()
    assert torch.equal(got, loss)
    _same(_state(layers), _state(ref))


def test_dz_of_a_pooled_layer_over_its_dy():
    """dz written where dy goes later, over the winners of the forward pass: the sums and gradients are those of a dz elsewhere."""
    import torch
    nf, ref, _, _, y = _block("bf16", 24, 21)
    nf, layers, _, _, _ = _block("bf16", 24, 21)
    R, L = ref[2], layers[2]
    x = torch.randn((24, 32, 32, 64), generator=torch.Generator(device="cuda").manual_seed(21), device="cuda").clamp_min(0).bfloat16()
    loss, act = torch.zeros(1, device="cuda"), R.new_act()
    R.set_skip_grad(torch.empty_like(L.stored("dy")))
    L.set_skip_grad(L.stored("dy"))
    for _ in range(2):
        R.step(x, y, 0.05, loss, act)
        L.step(x, y, 0.05, loss, act)
    torch.cuda.synchronize()
    _same(_state(layers), _state(ref))
