"""bf16 layers on maps that no 128-pixel tile divides: their convolutions once ran as fp32 chains on the CUDA cores, and the
tensor-core kernels that take them must not be further from the exact result than such chains are.  The yardstick is the library's own
fp32 convolution on the same bf16-valued operands (products of two bf16 numbers are exact in fp32): its error against 64 bits for the
fp32 weight gradients, and, for results that are rounded to bf16, the number of outputs whose rounding it gets wrong."""
import numpy as np
import pytest

from tests import parity_util as pu

pytestmark = pytest.mark.gpu

CASES = [  # every form: kernels of 64 and 128 output channels, one, two and four chunks of input channels, 16 to 128 filters, a pool, stride 2
    dict(N=61, Cin=256, Cout=256, H=14, W=14, F=16, classes=10, stride=1, pool=False),
    dict(N=61, Cin=128, Cout=256, H=28, W=28, F=32, classes=10, stride=2, pool=False),
    dict(N=200, Cin=64, Cout=256, H=14, W=14, F=64, classes=10, stride=1, pool=False),
    dict(N=160, Cin=64, Cout=64, H=14, W=22, F=24, classes=10, stride=1, pool=True),
    dict(N=1500, Cin=64, Cout=64, H=7, W=5, F=128, classes=10, stride=1, pool=False),
    dict(N=40, Cin=64, Cout=64, H=7, W=7, F=16, classes=10, stride=1, pool=False),       # small: weight gradients only on the tensor cores
    dict(N=12, Cin=64, Cout=64, H=56, W=56, F=16, classes=10, stride=1, pool=False),     # a size that the folded kernels would take
]


def _nhwc64(torch, x, w, stride):
    """Convolution of x [N,H,W,Ci] with w [9,Co,Ci] in 64 bits, [N,Ho,Wo,Co]."""
    out = []
    for a in x.split(max(1, (1 << 25) // (x[0].numel() * 9))):
        n, h, wd, c = a.shape
        u = torch.nn.functional.unfold(a.permute(0, 3, 1, 2).double(), 3, padding=1, stride=stride)       # [n, c*9, pixels]
        k = w.double().permute(1, 2, 0).reshape(w.shape[1], -1)
        out.append((k @ u).permute(0, 2, 1).reshape(n, (h - 1) // stride + 1, (wd - 1) // stride + 1, -1))
    return torch.cat(out)


def _wgrad64(torch, x, g, stride):
    """[9,Co,Ci] in 64 bits."""
    tot = 0
    m = max(1, (1 << 25) // (x[0].numel() * 9))
    for a, b in zip(x.split(m), g.split(m)):
        u = torch.nn.functional.unfold(a.permute(0, 3, 1, 2).double(), 3, padding=1, stride=stride)
        tot = tot + torch.einsum("ncp,nkp->ck", b.reshape(b.shape[0], -1, b.shape[3]).permute(0, 2, 1).double(), u)
    return tot.reshape(g.shape[3], x.shape[3], 9).permute(2, 0, 1)


def _off(got, exact):
    """Outputs that are not the bf16 value nearest to the exact one."""
    return int((got.float() != exact.float().bfloat16().float()).sum())


def _no_worse(n, ref):
    """Two counts of rare events: n is not larger than ref beyond what counts of that size scatter (three standard deviations)."""
    return n <= ref + 3.0 * np.sqrt(n + ref)


@pytest.mark.parametrize("ci", range(len(CASES)))
def test_ragged_layer_is_as_exact_as_fp32_chains(ci):
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    c = CASES[ci]
    P, x, y = pu.seeded_case(c, 40 + ci, bf16=True)
    P["gamma"][:], P["beta"][:] = 1.0, 0.0
    L = pu.gpu_layer(nf, c, P, nf.NF_BF16)
    assert all(L.kernel_family(k) == "tcgen05" for k in (1, 3)) and L.kernel_family(6) == "stored"
    assert all((L.kernel_family(k) == "tcgen05") == (c["N"] * L.Ha * L.Wa >= 8192) for k in (0, 2))
    xd = pu.to_device_nhwc(torch, np.maximum(x, 0.0), 1)
    act = L.new_act()
    L.step(xd, torch.from_numpy(y).cuda(), 0.0, torch.zeros(1, device="cuda"), act)
    torch.cuda.synchronize()
    assert L.status() == 0
    kw = lambda k: torch.from_numpy(np.ascontiguousarray(P[k].transpose(2, 3, 0, 1).reshape(9, P[k].shape[0], -1))).float().cuda()
    W, Wa, ba = kw("W"), kw("Wa"), torch.from_numpy(P["ba"]).cuda()
    Y, H, DH, DA, DY = (L.stored(k)[..., :c["F"]] if k in ("h", "dh") else L.stored(k) for k in ("y", "h", "dh", "da", "dy"))

    def chain(src, w, stride):
        n, h, wd, _ = src.shape
        out = torch.empty((n, (h - 1) // stride + 1, (wd - 1) // stride + 1, w.shape[1]), device="cuda")
        nf.nf_conv3x3_forward(nf.NF_F32, src.float().contiguous(), w.contiguous(), stride, out)
        return out

    # main forward, aux forward, aux input gradient
    e = _nhwc64(torch, xd, W, c["stride"])
    assert _no_worse(_off(Y, e), _off(chain(xd, W, c["stride"]).bfloat16(), e)), "y"
    e = (_nhwc64(torch, act, Wa, 1) + ba.double()).clamp_min(0)
    assert _no_worse(_off(H, e), _off((chain(act, Wa, 1) + ba).clamp_min(0).bfloat16(), e)), "h"
    wt = Wa.flip(0).permute(0, 2, 1).contiguous()
    e = _nhwc64(torch, DH, wt, 1)
    assert _no_worse(_off(DA, e), _off(chain(DH, wt, 1).bfloat16(), e)), "da"
    # weight gradients
    for name, src, g, stride in (("W", xd, DY, c["stride"]), ("Wa", act, DH, 1)):
        e = _wgrad64(torch, src, g, stride)
        got = torch.from_numpy(np.ascontiguousarray(L.get_param(name, nf.NF_K_GRAD).transpose(2, 3, 0, 1))).cuda().reshape(e.shape)
        ref = torch.empty(e.shape, device="cuda")
        s, gf = src.float().contiguous(), g.float().contiguous()
        n = nf.nf_conv3x3_wgrad_scratch_bytes(*s.shape, gf.shape[3], stride)
        nf.nf_conv3x3_wgrad(nf.NF_F32, s, gf, stride, torch.empty(n, dtype=torch.uint8, device="cuda"), ref)
        err = lambda t: float((t.double() - e).norm() / e.norm())
        assert err(got) <= err(ref), (name, err(got), err(ref))
    # statistics and BatchNorm-backward sums: fp32 chains of some tens of pixels, finished in 64 bits -- a few units of 2^-24
    y64 = Y.double()
    m, v = y64.mean((0, 1, 2)), y64.var((0, 1, 2), unbiased=False)
    cnt = y64.numel() // c["Cout"]
    rm, rv = (torch.from_numpy(L.get_param(k)).cuda().double() for k in ("rmean", "rvar"))
    assert float((rm / 0.1 - m).abs().max()) <= 8 * 2.0 ** -24 * float(v.sqrt().max() + m.abs().max())
    assert float(((rv - 0.9) / 0.1 * (cnt - 1) / cnt / v - 1).abs().max()) <= 0.9 / 0.1 * 2.0 ** -23 / float(v.min()) + 16 * 2.0 ** -24
    if not c["pool"]:
        xh = (y64 - m) / torch.sqrt(v + 1e-5)
        dz = torch.where(xh > 0, DA.double(), 0.0)
        e = (dz * xh).sum((0, 1, 2))
        got = torch.from_numpy(L.get_param("gamma", nf.NF_K_GRAD)).cuda().double()
        assert float((got - e).norm() / e.norm()) <= 4 * 2.0 ** -24, "ggamma"
    L.close()
