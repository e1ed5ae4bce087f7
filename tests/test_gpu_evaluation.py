"""Evaluation (nf_layer_predict, nf_block_cache): in place, on every form of the forward convolution."""
import numpy as np
import pytest

from paper_2402_14139_b200 import synth
from tests import parity_util as pu

pytestmark = pytest.mark.gpu


def _layer(nf, c, seed):
    """A layer of config c with weights and running statistics of its own."""
    P, x, _ = pu.seeded_case(c, seed, bf16=True)
    G = pu.gpu_layer(nf, c, P, nf.NF_BF16)
    rm = (0.2 * synth.normal(seed, 41, (c["Cout"],))).astype(np.float32)
    rv = (0.5 + synth.uniform01(seed, 42, c["Cout"])).astype(np.float32)
    G.set_param("rmean", rm)
    G.set_param("rvar", rv)
    return P, np.maximum(x, 0.0), rm, rv, G


IN_PLACE = [  # Cin = Cout, stride 1, no pool: the output has the input's shape
    dict(N=20, Cin=64, Cout=64, H=32, W=32, F=16, classes=10, stride=1, pool=False),    # folded column taps
    dict(N=70, Cin=64, Cout=64, H=16, W=16, F=16, classes=10, stride=1, pool=False),    # resident weights
    dict(N=70, Cin=128, Cout=128, H=16, W=16, F=16, classes=10, stride=1, pool=False),  # three boxes per chunk
    dict(N=90, Cin=256, Cout=256, H=8, W=8, F=16, classes=10, stride=1, pool=False),    # 256-wide, several images per tile
    dict(N=60, Cin=128, Cout=128, H=14, W=14, F=16, classes=10, stride=1, pool=False),  # segments
    dict(N=9, Cin=64, Cout=64, H=9, W=9, F=16, classes=10, stride=1, pool=False),       # CUDA cores
]


@pytest.mark.parametrize("ci", range(len(IN_PLACE)))
def test_evaluation_in_place(ci):
    """act_out = x, a cache that overlaps its input, and an output shifted against the input give what separate buffers give."""
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    c = IN_PLACE[ci]
    _, x, _, _, G = _layer(nf, c, 0x4E46F000 + ci)
    xd = pu.to_device_nhwc(torch, x, 1)
    want, pred, pred2 = G.new_act(), torch.zeros(c["N"], dtype=torch.int32, device="cuda"), torch.zeros(c["N"], dtype=torch.int32, device="cuda")
    G.predict(xd, pred, act_out=want)
    a = xd.clone()
    G.predict(a, pred2, act_out=a)
    assert torch.equal(a, want) and torch.equal(pred, pred2)
    blk = nf.Block([G])
    a = xd.clone()
    blk.cache(a, a)
    assert torch.equal(a, want)
    both = torch.zeros(xd.numel() + xd[0].numel(), dtype=torch.bfloat16, device="cuda")   # the output starts one image behind the input
    both[:xd.numel()] = xd.flatten()
    blk.cache(both[:xd.numel()], both[xd[0].numel():])
    assert torch.equal(both[xd[0].numel():], want.flatten())
    torch.cuda.synchronize()
    assert G.status() == 0
    blk.close()
    G.close()


FORMS = [  # (config, count): every instantiation that normalises in the convolution's epilogue, and the stride-2 ones
    (dict(N=9, Cin=64, Cout=64, H=32, W=32, F=16, classes=10, stride=1, pool=False), 7),     # folded column taps
    (dict(N=6, Cin=3, Cout=64, H=32, W=32, F=16, classes=10, stride=1, pool=False), 5),      # folded, input padded to 16 channels
    (dict(N=12, Cin=64, Cout=64, H=16, W=16, F=16, classes=10, stride=1, pool=False), 9),    # resident weights
    (dict(N=9, Cin=64, Cout=128, H=16, W=16, F=16, classes=10, stride=1, pool=False), 8),    # three boxes per chunk, 128 channels
    (dict(N=9, Cin=128, Cout=64, H=16, W=16, F=16, classes=10, stride=1, pool=False), 8),    # the same, 64 channels
    (dict(N=11, Cin=64, Cout=256, H=8, W=8, F=16, classes=10, stride=1, pool=False), 9),     # 256 channels in two halves
    (dict(N=11, Cin=64, Cout=128, H=8, W=8, F=16, classes=10, stride=1, pool=False), 9),     # per tap, 128 channels
    (dict(N=11, Cin=64, Cout=64, H=16, W=16, F=16, classes=10, stride=2, pool=False), 9),    # per tap, 64 channels
    (dict(N=45, Cin=64, Cout=128, H=14, W=14, F=16, classes=10, stride=1, pool=False), 43),  # segments, 128 channels
    (dict(N=12, Cin=64, Cout=64, H=28, W=28, F=16, classes=10, stride=1, pool=False), 11),   # segments, 64 channels
    (dict(N=45, Cin=64, Cout=256, H=14, W=14, F=16, classes=10, stride=1, pool=False), 11),  # fewer than 8192 pixels of a batch that has them
]


@pytest.mark.parametrize("ci", range(len(FORMS)))
def test_every_form_of_the_evaluating_convolution(ci):
    """predict and cache with running statistics against the checker, for fewer samples than the batch size; rows beyond are left alone."""
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    c, count = FORMS[ci]
    P, x, rm, rv, G = _layer(nf, c, 0x4E46F100 + ci)
    assert G.kernel_family(0) == "tcgen05"
    O = pu.oracle_layer(c, P, store_bf16=True)
    O.set(rmean=rm, rvar=rv)
    act_o, logits_o, _ = O.predict(x[:count])
    xd = pu.to_device_nhwc(torch, x[:count], 1)
    act, cache = G.new_act(), G.new_act()
    act.fill_(7.0)
    cache.fill_(7.0)
    logits, pred = torch.zeros((count, c["classes"]), device="cuda"), torch.zeros(count, dtype=torch.int32, device="cuda")
    G.predict(xd, pred, act_out=act, logits_out=logits, count=count)
    blk = nf.Block([G])
    blk.cache(xd, cache, count=count)
    torch.cuda.synchronize()
    assert G.status() == 0
    # stored twice in bf16 on both sides: a unit of 2^-8 of the value where the roundings of y fall on different sides
    err = np.abs(pu.from_device_nhwc(act)[:count] - act_o)
    assert (err <= 2.0 ** -7 * np.abs(act_o) + 2.0 ** -8 * np.abs(act_o).max()).all()
    assert (err > 2.0 ** -9 * np.abs(act_o).max()).mean() <= 0.01
    assert np.abs(logits.cpu().numpy() - logits_o).max() <= pu.TOL[1]["t"] * np.abs(logits_o).max()
    assert torch.equal(cache, act) and bool((act[count:] == 7.0).all())
    blk.close()
    G.close()
