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
