"""Timed cases of the local-layer training framework, over the sizes that its workloads have.

A case is a plain dict.  "kind" says which calls a pass makes, "net" and "block" which layers of
`paper_2402_14139_b200/workloads.py` it makes them on, "batch" the block's batch size:

  step      one Block.step on device tensors, launched kernel by kernel
  graph     the same step replayed from Block.capture
  host      one Block.step_host_next: the batch comes from pinned host memory, the losses go back
  stage     Block.step of a stage of an ImageNet-shaped residual network behind the c4 block (stride 2, then stride 1),
            whose map sizes are whatever the image size leaves
  residual  a CIFAR-100-shaped residual stage with its shortcuts: the projection, the trainable shortcut, the identity one
  exits     Layer.predict of every layer of a block on a part of a batch (early-exit evaluation)
  handover  Block.cache of a finished block, then nf_cache_gather of the next block's batch out of the cache

A training pass returns the losses, the block's output and every layer's gradients (all parameters of a layer in one
buffer).  The updated parameters and running statistics are what the next pass on the same state computes with.
"""
import math

import torch

from paper_2402_14139_b200 import nf, workloads

LR = 0.01


def listed():
    return [
        # one small fp32 layer on a handful of images: the least a call can be, all launches and latency
        dict(name="c1_step_fp32", kind="step", net="c1", block=0, batch=8),
        # the CIFAR-10-shaped VGG block at its own batch size, called from an ordinary training loop
        dict(name="c2_step", kind="step", net="c2", block=0, batch=128),
        # the same block fed from a data loader's pinned buffers, one batch ahead
        dict(name="c2_host", kind="host", net="c2", block=0, batch=128),
        # first stage of the CIFAR-100-shaped ResNet stack, recorded once and replayed
        dict(name="c3_stage1_graph", kind="graph", net="c3", block=0, batch=64),
        # second stage as the residual network has it, shortcuts included
        dict(name="c3_residual2", kind="residual", net="c3", block=1, batch=128),
        # the ImageNet-shaped block: few wide-open maps, the benchmark's workload
        dict(name="c4_step", kind="step", net="c4", block=0, batch=64),
        # what follows it in such a network: 28x28 -> 14x14 maps, more channels, a last batch of an odd size
        dict(name="imagenet_stage14", kind="stage", channels=256, size=28, batch=61),
        # Tiny-ImageNet-shaped VGG-16, second block: 64 channels with a max-pool, batch size as Algorithm 1 sets it
        dict(name="c5_block2_pool", kind="step", net="c5", block=1, batch=1904),
        # its last block: seven layers of 256 and 512 channels down to 2x2 maps at a very large batch
        dict(name="c5_block5", kind="step", net="c5", block=4, batch=8602),
        # wide auxiliary networks (256 filters), as the paper's filter rule gives them
        dict(name="c6_block3_wide_aux", kind="step", net="c6", block=2, batch=6366),
        # early-exit evaluation of a trained block on the rest of a validation set
        dict(name="c5_exits4", kind="exits", net="c5", block=3, batch=2048, count=1777),
        # a block has finished: its outputs go to the cache, and the next block's first batch comes out of it
        dict(name="c5_handover1", kind="handover", net="c5", block=0, batch=1260, take=952),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same kinds: other blocks of the workloads, batch sizes (odd ones too) up to the listed ones."""
    kind = rng.choice(["step"] * 5 + ["host", "graph", "residual", "stage", "stage", "exits", "handover"])
    if kind == "step":
        net, block, lo, hi = rng.choice([("c1", 0, 8, 512), ("c2", 0, 32, 512), ("c4", 0, 4, 64), ("c5", 0, 64, 1260), ("c5", 1, 64, 1904),
                                         ("c5", 2, 128, 3045), ("c5", 3, 256, 5935), ("c5", 4, 256, 8602), ("c6", 1, 128, 3452),
                                         ("c6", 2, 256, 6366), ("c6", 3, 512, 8192)])
        return dict(kind=kind, net=net, block=block, batch=_log(rng, lo, hi))
    if kind == "host":
        return dict(kind=kind, net="c2", block=0, batch=_log(rng, 32, 512))
    if kind == "graph":
        return dict(kind=kind, net="c3", block=rng.randrange(4), batch=_log(rng, 48, 768))
    if kind == "residual":
        return dict(kind=kind, net="c3", block=rng.randrange(1, 4), batch=_log(rng, 48, 512))
    if kind == "stage":
        k = rng.randrange(3)  # images of 96 to 256 pixels: each stage halves the maps and doubles the channels
        return dict(kind=kind, channels=128 << k, size=(rng.randint(96, 256) - 1) // (4 << k) + 1, batch=_log(rng, 16, 96))
    if kind == "exits":
        n = _log(rng, 128, 2048)
        return dict(kind=kind, net=rng.choice(["c5", "c6"]), block=rng.randrange(1, 5), batch=n, count=rng.randint(n // 2, n))
    n = _log(rng, 128, 1260)
    return dict(kind=kind, net="c5", block=rng.randrange(5), batch=n, take=rng.randint(n // 4, n))


def _layers(case):
    """(layer dicts, number of classes, dtype name) of a case."""
    if case["kind"] == "stage":
        c, s = case["channels"], case["size"]
        t = (s - 1) // 2 + 1
        return [dict(Cin=c // 2, Cout=c, H=s, W=s, F=16, stride=2, pool=False),
                dict(Cin=c, Cout=c, H=t, W=t, F=16, stride=1, pool=False)], 1000, "bf16"
    wl = workloads.ALL[case["net"]]()
    return wl["blocks"][case["block"]][1], wl["classes"], wl["dtype"]


def _build(case, gen):
    """nf.Layer objects with Kaiming-normal weights and the statistics of a layer in training."""
    specs, classes, dtype = _layers(case)
    made = []
    for i, l in enumerate(specs):
        L = nf.Layer(l["Cin"], l["Cout"], l["H"], l["W"], l["F"], classes, case["batch"], stride=l["stride"], maxpool=l["pool"],
                     dtype=nf.NF_F32 if dtype == "f32" else nf.NF_BF16, host_io=2 if case["kind"] == "host" and i == 0 else 0)
        for name, fan_in in (("W", 9 * l["Cin"]), ("Wa", 9 * l["Cout"]), ("Wf", 4 * l["F"])):
            w = torch.randn(L.shapes[name], generator=gen, device="cuda") * math.sqrt(2.0 / fan_in)
            L.set_param(name, w.cpu().numpy())
        if case["kind"] in ("exits", "handover"):
            L.set_param("rmean", (0.1 * torch.randn(l["Cout"], generator=gen, device="cuda")).cpu().numpy())
            L.set_param("rvar", (0.5 + 2.0 * torch.rand(l["Cout"], generator=gen, device="cuda")).cpu().numpy())
        made.append(L)
    return made


def _inputs(case, layers, gen, count=None):
    """A batch: normalised images for a first block (3 channels), activations after a ReLU for a later one; labels."""
    L, n = layers[0], count or case["batch"]
    x = torch.randn((n, L.H, L.W, L.Cin), generator=gen, device="cuda", dtype=torch.float32)
    if L.Cin > 3:
        x.clamp_(min=0)
    y = torch.randint(0, L.classes, (n,), generator=gen, device="cuda", dtype=torch.int32)
    return x.to(L.tdtype), y


def prepare(case, seed):
    nf.nf_set_stream(torch.cuda.current_stream())
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    layers = _build(case, gen)
    x, y = _inputs(case, layers, gen)
    s = dict(kind=kind, layers=layers, x=x, y=y, grads=[L.dp_buffer(2) for L in layers],
             loss=torch.zeros(len(layers), device="cuda"))
    if kind == "residual":
        b, L = layers[0], layers[1]
        p = nf.Projection(b.Cin, L.Cout, b.H, b.W, case["batch"])
        p.set_param("W", (torch.randn(p.shapes["W"], generator=gen, device="cuda") * math.sqrt(1.0 / b.Cin)).cpu().numpy())
        s.update(proj=p, short=p.new_out(), dz=p.new_out(), acts=[L.new_act() for L in layers])
        L.set_skip(s["short"])
        L.set_skip_grad(s["dz"])
        layers[3].set_skip(s["acts"][1])
        s["losses"] = [s["loss"][i:i + 1] for i in range(4)]
        return s
    if kind == "exits":
        n = case["count"]
        s.update(count=n, x=x[:n].contiguous(), acts=[L.new_act()[:n] for L in layers],
                 logits=[torch.empty((n, L.classes), device="cuda") for L in layers],
                 pred=[torch.empty(n, dtype=torch.int32, device="cuda") for L in layers])
        return s
    s["block"] = nf.Block(layers)
    last = layers[-1]
    if kind == "handover":
        s.update(cache=torch.empty((case["batch"], last.Ha, last.Wa, last.Cout), dtype=last.tdtype, device="cuda"),
                 idx=torch.randperm(case["batch"], generator=gen, device="cuda")[:case["take"]].to(torch.int32))
        s.update(out=torch.empty_like(s["cache"][:case["take"]]), out_y=torch.empty(case["take"], dtype=torch.int32, device="cuda"))
        return s
    s["act"] = last.new_act()
    if kind == "host":
        more = _inputs(case, layers, gen)
        s["batches"] = [(a.cpu().pin_memory(), b.cpu().pin_memory()) for a, b in ((x, y), more)]
        s["loss"], s["turn"] = torch.zeros(len(layers)).pin_memory(), 0
    if kind == "graph":
        s["block"].step(x, y, LR, s["loss"], s["act"])
        s["graph"] = s["block"].capture(x, y, LR, s["loss"], s["act"])
    return s


def run(s):
    kind = s["kind"]
    if kind in ("step", "stage"):
        s["block"].step(s["x"], s["y"], LR, s["loss"], s["act"])
        return dict(loss=s["loss"], act=s["act"], grads=s["grads"])
    if kind == "graph":
        s["graph"].replay()
        return dict(loss=s["loss"], act=s["act"], grads=s["grads"])
    if kind == "host":
        (x, y), (nx, ny) = s["batches"][s["turn"]], s["batches"][1 - s["turn"]]
        s["block"].step_host_next(x, y, LR, s["loss"], nx, ny)
        s["turn"] = 1 - s["turn"]
        return dict(loss=s["loss"], grads=s["grads"])
    if kind == "residual":
        a, (l0, l1, l2, l3), e = s["acts"], s["layers"], s["losses"]
        s["proj"].forward(s["x"], s["short"])
        l0.step(s["x"], s["y"], LR, e[0], a[0])
        l1.step(a[0], s["y"], LR, e[1], a[1])
        s["proj"].backward(s["x"], s["dz"], LR)
        l2.step(a[1], s["y"], LR, e[2], a[2])
        l3.step(a[2], s["y"], LR, e[3], a[3])
        return dict(loss=s["loss"], act=a[3], short=s["short"], dz=s["dz"], grads=s["grads"])
    if kind == "exits":
        x = s["x"]
        for L, act, logits, pred in zip(s["layers"], s["acts"], s["logits"], s["pred"]):
            L.predict(x, pred, act_out=act, logits_out=logits, count=s["count"])
            x = act
        return dict(act=x, logits=s["logits"], pred=s["pred"])
    s["block"].cache(s["x"], s["cache"])
    nf.nf_cache_gather(s["cache"], s["y"], s["idx"], s["out"], s["out_y"])
    return dict(cache=s["cache"], rows=s["out"], labels=s["out_y"])


def work(case):
    """Per layer: its input is read and its output written; a training step also reads and writes parameters and momentum and
    writes the gradients.  Arithmetic: the two convolutions in each direction they are needed in, and the linear layer."""
    specs, classes, dtype = _layers(case)
    es, n = (4 if dtype == "f32" else 2), case.get("count", case["batch"])
    train = case["kind"] not in ("exits", "handover")
    total, flops = 0.0, 0.0
    for l in specs:
        ha, wa = workloads.out_hw(l)
        f = workloads.step_flops(l, n)
        main, aux = 9 * l["Cin"] * l["Cout"] + 2 * l["Cout"], 9 * l["Cout"] * l["F"] + l["F"] + classes * (4 * l["F"] + 1)
        total += es * n * (l["H"] * l["W"] * l["Cin"] + ha * wa * l["Cout"])
        if case["kind"] == "handover":
            total, flops = total + es * main, flops + f["conv_fwd"]
        elif train:
            total += (main + aux) * 20 + 4 * n
            flops += f["conv_fwd"] + f["wgrad"] + f["aux_fwd"] + f["aux_bwd"] + 3 * 2.0 * n * 4 * l["F"] * classes
        else:
            total += (main + aux) * es + 4 * n * (classes + 1)
            flops += f["conv_fwd"] + f["aux_fwd"] + 2.0 * n * 4 * l["F"] * classes
    if case["kind"] == "handover":
        ha, wa = workloads.out_hw(specs[-1])
        total += case["take"] * (2 * es * ha * wa * specs[-1]["Cout"] + 12)
    if case["kind"] == "residual":
        l = specs[0]
        ho, wo = workloads.out_hw(l)
        flops += 2 * 2.0 * n * ho * wo * l["Cin"] * l["Cout"]
        total += es * n * ho * wo * (l["Cin"] + 2 * l["Cout"]) + 20 * l["Cin"] * l["Cout"]
    return dict(bytes=total, flops=flops)


def tolerance(case):
    """fp32: sums over a batch in another order.  bf16: activations are stored in bf16, and where two summation orders straddle
    a rounding boundary a ReLU or a max-pool decides differently now and then, which moves a gradient by about 1%; without
    gradients only the roundings remain.  Classes change where the two largest logits are as close as that."""
    if _layers(case)[2] == "f32":
        return dict(rel=2e-5)
    if case["kind"] == "handover":
        return dict(rel=5e-3)
    if case["kind"] == "exits":
        return dict(rel=5e-3, differ=0.01)
    return dict(rel=2e-2)
