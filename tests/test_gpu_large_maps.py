"""More output pixels than 31 bits number: the CUDA-core convolution and the projection."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 70000, 31000), (3, 28000, 26000)])  # rows of one image per launch; two images, then one
def test_convolution_of_more_than_2_31_pixels(shape):
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    N, H, W = shape
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = torch.empty((N, H, W, 1), dtype=torch.bfloat16, device="cuda")
    for n in range(N):
        for h in range(0, H, 8192):      # small whole numbers: every sum is exact
            x[n, h:h + 8192] = torch.randint(-2, 3, x[n, h:h + 8192].shape, generator=g, device="cuda", dtype=torch.int8).to(torch.bfloat16)
    w = torch.tensor([1, -2, 1, 2, -1, 1, -2, 2, -1], device="cuda").to(torch.bfloat16).reshape(9, 1, 1)
    y = torch.full((N, H, W, 1), float("nan"), dtype=torch.bfloat16, device="cuda")
    nf.nf_conv3x3_forward(nf.NF_BF16, x, w, 1, y)
    torch.cuda.synchronize()
    split = (2 ** 31 - 1) // W           # first row of the second launch, where an image takes two
    for n in range(N):
        for a, b in ((0, 3), (split - 2, split + 2), (H // 2, H // 2 + 2), (H - 3, H)):
            if not 0 < a < H or b > H:
                a, b = 0, 3
            lo, hi = max(a - 1, 0), min(b + 1, H)
            xs = torch.nn.functional.pad(x[n, lo:hi, :, 0].float(), (1, 1, 0 if lo < a else 1, 0 if hi > b else 1))
            want = sum(w[3 * i + j].float().item() * xs[i:i + b - a, j:j + W] for i in range(3) for j in range(3))
            assert torch.equal(y[n, a:b, :, 0].float(), want), (n, a)
    assert not any(bool(y[n].isnan().any()) for n in range(N))


def test_projection_of_more_than_2_31_pixels():
    """The second input channel has zero weight and is 1 at one output pixel near the end: its weight gradient is the gradient there."""
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    S = 46400
    GP = nf.Projection(2, 1, 2 * S, 2 * S, 1, bn_momentum=1.0)
    GP.set_param("W", np.array([[0.5, 0.0]], dtype=np.float32))
    xb = torch.zeros((1, 2 * S, 2 * S, 2), dtype=torch.bfloat16, device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    for h in range(0, 2 * S, 8192):
        xb[0, h:h + 8192, :, 0] = torch.randint(-8, 9, xb[0, h:h + 8192, :, 0].shape, generator=g, device="cuda", dtype=torch.int8).to(torch.bfloat16)
    i, j = S - 3, S - 5
    assert i * S + j > 2 ** 31
    xb[0, 2 * i, 2 * j, 0] = 3.0
    xb[0, 2 * i, 2 * j, 1] = 1.0
    s, dz = GP.new_out(), GP.new_out()
    GP.forward(xb, s)
    dz.fill_(1.0)
    dz[0, i, j] = 4.0
    dz[0, : S // 2] = -0.5
    GP.backward(xb, dz, 0.0)
    torch.cuda.synchronize()
    M = float(S) * S
    mu, var = float(GP.get_param("rmean")[0]), float(GP.get_param("rvar")[0])
    m1, m2 = (float(GP.get_param(k, nf.NF_K_GRAD)[0]) / M for k in ("beta", "gamma"))
    inv = 1.0 / np.sqrt(var + 1e-5)
    want_s = (1.5 - mu) * inv
    want = inv * (4.0 - m1 - want_s * m2)
    assert abs(mu) < 0.01 and abs(var - 6.0) < 0.01 and abs(m1 - 0.25) < 1e-3      # variance of 0.5 * (-8 .. 8)
    assert abs(float(s[0, i, j, 0]) - want_s) <= 2.0 ** -8 * abs(want_s)
    assert abs(float(GP.get_param("W", nf.NF_K_GRAD)[0, 1]) - want) <= 2.0 ** -8 * abs(want)
    GP.close()
