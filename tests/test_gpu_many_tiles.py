"""Kernels that walk many tiles per block: every ring and buffer of theirs is used again and again, which the smaller parity shapes (one
or two tiles per block) do not reach.  Each result of a step is compared with a 64-bit computation from the step's own stored inputs."""
import numpy as np
import pytest

from tests import parity_util as pu
from tests.test_gpu_ragged_precision import _nhwc64, _wgrad64

pytestmark = pytest.mark.gpu

# B200: 148 blocks.  tiles of 128 pixels x channel tiles per block, and what is used again
CASES = [
    # 596 tiles of 256 channels (4 per block): halves leave through one staging tile, statistics per half; the input gradient of 16
    # filters has 1192 tiles (8 per block): two staging and two y slots handed to the summing group; the last image group is half empty
    dict(N=1191, Cin=64, Cout=256, H=8, W=8, F=16, classes=10, stride=1, pool=False),
    # the input gradient of 256 filters: 256-wide, y tiles loaded by the epilogue, half by half
    dict(N=1191, Cin=64, Cout=256, H=8, W=8, F=256, classes=10, stride=1, pool=False),
    # eight images per tile, the last group with three of them; 128 and 64 channels per tile
    dict(N=4739, Cin=64, Cout=128, H=4, W=4, F=8, classes=10, stride=1, pool=False),
    dict(N=4739, Cin=64, Cout=64, H=4, W=4, F=8, classes=10, stride=1, pool=False),
    # segments: four accumulators in turn, weight gradient pairs of segments (many tiles per split), tiles over the edges
    dict(N=700, Cin=64, Cout=128, H=14, W=14, F=16, classes=10, stride=1, pool=False),
    dict(N=700, Cin=128, Cout=64, H=14, W=14, F=40, classes=10, stride=1, pool=False),
]


@pytest.mark.parametrize("ci", range(len(CASES)))
def test_step_with_many_tiles_per_block(ci):
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    c = CASES[ci]
    P, x, y = pu.seeded_case(c, 1400 + ci, bf16=True)
    P["gamma"][:], P["beta"][:] = 1.0, 0.0
    L = pu.gpu_layer(nf, c, P, nf.NF_BF16)
    assert all(L.kernel_family(k) == "tcgen05" for k in range(4)) and L.kernel_family(6) == "stored"
    xd, act = pu.to_device_nhwc(torch, np.maximum(x, 0.0), 1), L.new_act()
    for _ in range(2):          # the second step finds the barriers' memory and the workspace used
        L.step(xd, torch.from_numpy(y).cuda(), 0.0, torch.zeros(1, device="cuda"), act)
    torch.cuda.synchronize()
    assert L.status() == 0
    kw = lambda k: torch.from_numpy(np.ascontiguousarray(P[k].transpose(2, 3, 0, 1).reshape(9, P[k].shape[0], -1))).float().cuda()
    W, Wa, ba = kw("W"), kw("Wa"), torch.from_numpy(P["ba"]).cuda().double()
    Y, H, DH, DA, DY = (L.stored(k)[..., :c["F"]] if k in ("h", "dh") else L.stored(k) for k in ("y", "h", "dh", "da", "dy"))

    def rounded(got, exact, what):      # bf16 keeps 8 bits: half a unit is at most 2^-8 of a value; sums in fp32 add 2^-12 of the largest
        lim = 2.0 ** -8 * exact.abs() + 2.0 ** -12 * exact.abs().max()
        assert bool(((got.double() - exact).abs() <= lim).all()), what

    rounded(Y, _nhwc64(torch, xd, W, 1), "y")
    rounded(H, (_nhwc64(torch, act, Wa, 1) + ba).clamp_min(0), "h")
    rounded(DA, _nhwc64(torch, DH, Wa.flip(0).permute(0, 2, 1).contiguous(), 1), "da")
    y64 = Y.double()
    m, v = y64.mean((0, 1, 2)), y64.var((0, 1, 2), unbiased=False)
    xh = (y64 - m) / torch.sqrt(v + 1e-5)
    rounded(act, xh.clamp_min(0), "act")
    dz = torch.where(xh > 0, DA.double(), 0.0)
    sums = dict(beta=dz.sum((0, 1, 2)), gamma=(dz * xh).sum((0, 1, 2)))
    near = lambda got, exact, what: _near(torch, got, exact, what)
    for k, e in sums.items():
        near(L.get_param(k, nf.NF_K_GRAD), e, "g" + k)
    M = y64.numel() // c["Cout"]
    rounded(DY, (dz - sums["beta"] / M - xh * sums["gamma"] / M) / torch.sqrt(v + 1e-5), "dy")
    for name, src, g in (("W", xd, DY), ("Wa", act, DH)):
        e = _wgrad64(torch, src, g, 1)
        near(np.ascontiguousarray(L.get_param(name, nf.NF_K_GRAD).transpose(2, 3, 0, 1)).reshape(e.shape), e, "g" + name)
    near(L.get_param("ba", nf.NF_K_GRAD), DH.double().sum((0, 1, 2)), "gba")
    L.close()


def _near(torch, got, exact, what):
    """fp32 sums over up to 137 000 pixels, a few of which change sides of the ReLU with the rounding of the statistics: 1e-3 of the size;
    a tile lost or taken twice would be 1 / (tiles) or more, 4e-3 of 296 tiles' random sums at the least times its square root."""
    e = exact.cpu().numpy()
    assert np.sqrt(((got - e) ** 2).sum() / (e ** 2).sum()) <= 1e-3, what
