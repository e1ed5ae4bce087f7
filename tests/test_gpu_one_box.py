"""Auxiliary forward and input gradient without sums over their tiles (one activation box per chunk, two epilogue groups) and the average
pool in one pass: every instantiation, with tiles left over at the end of a block's range, against 64 bits from the layer's own tensors."""
import numpy as np
import pytest

from tests import parity_util as pu
from tests.test_gpu_ragged_precision import _nhwc64, _wgrad64

pytestmark = pytest.mark.gpu


def _c(N, Cout, H, W, F, pool=False, da=True):
    """A case; `da`: whether the layer stores da (else its input gradient runs twice and only its sums and dy leave it)."""
    return dict(N=N, Cin=64, Cout=Cout, H=H, W=W, F=F, classes=10, stride=1, pool=pool), da


CASES = [
    # aux forward with 64 filters: two groups in turn, odd numbers of tiles per block; one chunk (resident weights) and two
    _c(75, 64, 32, 32, 64), _c(41, 128, 32, 16, 64), _c(1, 64, 16, 8, 64),
    # one box per chunk, weights resident / in the stages: 16 filters over four and eight chunks, 32 over two and four; 40 filters: in 64 columns
    _c(77, 256, 16, 16, 16, da=False), _c(37, 512, 16, 16, 16, da=False), _c(77, 128, 16, 16, 32, da=False), _c(39, 256, 16, 16, 24, da=False),
    _c(21, 128, 16, 16, 40),
    # pooled layers: input gradient of 16, 32 and 64 filters to 128 and 64 channels, one box, two groups
    _c(77, 128, 32, 32, 16, True), _c(39, 128, 32, 32, 32, True), _c(150, 64, 64, 64, 64, True), _c(151, 64, 32, 16, 16, True), _c(75, 64, 32, 16, 32, True),
    # maps 8 pixels wide: weight gradient of 16, 32 and 64 filters from one box per tile, the last tile short of images
    _c(75, 128, 8, 8, 16), _c(2, 64, 8, 8, 32), _c(77, 64, 4, 8, 64), _c(1203, 64, 8, 8, 8),
    # many images: the head pools (chains of one, two and eight pixels), or the kernel for 8x8 with 256 filters (a division at the end)
    _c(1500, 64, 16, 16, 8, da=False), _c(300, 64, 32, 32, 16, da=False), _c(1000, 64, 32, 32, 64), _c(700, 64, 8, 8, 256), _c(170, 64, 20, 20, 8),
]


def _check_pool(torch, L, N, F):
    H = L.stored("h")[:N, ..., :F]
    ha, wa = H.shape[1] // 2, H.shape[2] // 2
    p64 = torch.stack([H[:, a * ha:(a + 1) * ha, b * wa:(b + 1) * wa].double().mean((1, 2)) for a in (0, 1) for b in (0, 1)], -1)
    p = L.stored("p")[:N].view(N, -1, 4)[:, :F]
    # fp32 sums of up to 256 values of one sign: at most 256 half units of 2^-24 each
    assert bool(((p.double() - p64).abs() <= 2.0 ** -16 * p64 + 1e-7).all()), "p"


@pytest.mark.parametrize("ci", range(len(CASES)))
def test_forms_without_sums(ci):
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    c, da = CASES[ci]
    P, x, y = pu.seeded_case(c, 2600 + ci, bf16=True)
    L = pu.gpu_layer(nf, c, P, nf.NF_BF16)
    xd, act = pu.to_device_nhwc(torch, np.maximum(x, 0.0), 1), L.new_act()
    for _ in range(2):
        L.step(xd, torch.from_numpy(y).cuda(), 0.0, torch.zeros(1, device="cuda"), act)
    torch.cuda.synchronize()
    assert L.status() == 0
    F = c["F"]
    Wa = torch.from_numpy(np.ascontiguousarray(P["Wa"].transpose(2, 3, 0, 1).reshape(9, F, -1))).float().cuda()
    h = (_nhwc64(torch, act, Wa, 1) + torch.from_numpy(P["ba"]).cuda().double()).clamp_min(0)

    def rounded(got, exact, what):      # bf16 keeps 8 bits: half a unit is at most 2^-8 of a value; sums in fp32 add 2^-12 of the largest
        lim = 2.0 ** -8 * exact.abs() + 2.0 ** -12 * exact.abs().max()
        assert bool(((got.double() - exact).abs() <= lim).all()), what

    assert [L.kernel_family(k) for k in (0, 1, 2, 3, 7)] == ["tcgen05"] * 5
    assert L.kernel_family(5) == "stored" and L.kernel_family(6) == ("stored" if da else "two-pass")
    rounded(L.stored("h")[..., :F], h, "h")
    _check_pool(torch, L, c["N"], F)
    if da:
        rounded(L.stored("da"), _nhwc64(torch, L.stored("dh")[..., :F], Wa.flip(0).permute(0, 2, 1).contiguous(), 1), "da")
    if not c["pool"]:
        g64 = _wgrad64(torch, act, L.stored("dh")[..., :F], 1).cpu().numpy()
        g = np.ascontiguousarray(L.get_param("Wa", nf.NF_K_GRAD).transpose(2, 3, 0, 1)).reshape(g64.shape)
        # exact products; the running sum of the tensor core loses 2^-27 per instruction, a few hundred of them per range
        assert np.sqrt(((g - g64) ** 2).sum() / (g64 ** 2).sum()) <= 1e-5, "gWa"
    L.close()


# (images, map, filters, kernels of the pool): one pass with chains of one pixel (64, 256 and 100 of them), two, four and eight pixels; the two
# kernels below the lines between; 4x4 and 8x8 maps with a division at the end
POOLS = [(1500, 16, 8, 1), (4097, 32, 8, 1), (2049, 20, 16, 1), (1537, 16, 64, 1), (3073, 32, 32, 1), (1537, 32, 64, 1), (385, 16, 256, 1),
         (4095, 32, 8, 2), (1535, 16, 64, 2), (700, 8, 256, 1), (19000, 4, 8, 1)]


@pytest.mark.parametrize("N,S,F,kernels", POOLS)
def test_average_pool_of_an_evaluation(N, S, F, kernels):
    """An exit pools h with kernels of its own."""
    import torch
    from paper_2402_14139_b200 import nf
    nf.nf_set_stream(torch.cuda.current_stream())
    gen = torch.Generator(device="cuda").manual_seed(N)
    L = nf.Layer(8, 8, S, S, F, 10, N)
    for name in ("W", "Wa", "Wf"):
        L.set_param(name, (0.2 * torch.randn(L.shapes[name], generator=gen, device="cuda")).cpu().numpy())
    x = torch.randn((N, S, S, 8), generator=gen, device="cuda").bfloat16()
    before = nf.nf_launch_count()
    L.predict(x, torch.empty(N, dtype=torch.int32, device="cuda"))
    # coefficients, convolution, BatchNorm, auxiliary convolution, pool, head (one kernel, for many images three)
    assert nf.nf_launch_count() - before == 4 + kernels + (3 if N * 4 * F * 10 >= 1 << 24 else 1)
    _check_pool(torch, L, N, F)
    L.close()
