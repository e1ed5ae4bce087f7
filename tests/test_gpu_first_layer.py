"""Evaluation of an RGB first layer straight from the images: against 64 bits, at the edges of tiles and images, and where the output
overlaps the images (the padded copy stays in use there)."""
import pytest

pytestmark = pytest.mark.gpu

# (N, count, H, W): tiles of 16 x 8 and 8 x 16 pixels, one tile per image, more tiles than three blocks per SM take, fewer images than N
SHAPES = [(1, 1, 8, 32), (3, 3, 16, 40), (5, 2, 32, 32), (2, 2, 48, 112), (97, 90, 32, 64), (2, 2, 224, 224)]


def _layer(N, H, W, seed):
    import torch
    from paper_2402_14139_b200 import nf
    nf.nf_set_stream(torch.cuda.current_stream())
    gen = torch.Generator(device="cuda").manual_seed(seed)
    L = nf.Layer(3, 64, H, W, 16, 10, N)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    p = dict(W=rnd(64, 3, 3, 3) * (2 / 27) ** 0.5, gamma=1 + 0.2 * rnd(64), beta=0.3 * rnd(64), rmean=0.1 * rnd(64), rvar=0.5 + 2 * rnd(64).abs())
    for k, v in p.items():
        L.set_param(k, v.cpu().numpy())
    return nf, L, p, rnd(N, H, W, 3).bfloat16()


def _reference(x, p):
    """(act, y * scale) in 64 bits from the stored inputs and bf16 weights."""
    import torch
    y = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), p["W"].bfloat16().double(), padding=1).permute(0, 2, 3, 1)
    s = p["gamma"].double() / torch.sqrt(p["rvar"].double() + 1e-5)
    return (y * s + (p["beta"].double() - p["rmean"].double() * s)).clamp_min(0), y * s


def _cache(nf, block, x, out, launches, count=None):
    """Block.cache, with the number of its launches: 2 straight from the images (coefficients, convolution), 4 by way of padded copies of
    the images and the weights."""
    before = nf.nf_launch_count()
    block.cache(x, out, count=count)
    assert nf.nf_launch_count() - before == launches


def _check(got, want, ys):
    # y and the result are rounded to 8 bits each: half a unit is at most 2^-8 of the value; 27 products in fp32 are far below that
    assert bool(((got.double() - want).abs() <= 2.0 ** -8 * (ys.abs() + want) + 1e-5).all())


@pytest.mark.parametrize("N,count,H,W", SHAPES)
def test_first_layer_against_64_bits(N, count, H, W):
    import torch
    nf, L, p, x = _layer(N, H, W, H + W)
    out = torch.full((N, H, W, 64), 7.0, dtype=torch.bfloat16, device="cuda")
    _cache(nf, nf.Block([L]), x, out, 2, count)
    _check(out[:count], *_reference(x[:count], p))
    assert bool((out[count:] == 7.0).all()) and L.status() == 0


def test_images_with_infinities_reach_their_neighbours_only():
    import torch
    nf, L, p, x = _layer(2, 32, 32, 5)
    out, ref = (torch.empty((2, 32, 32, 64), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    block = nf.Block([L])
    _cache(nf, block, x, ref, 2)
    for r, c in ((0, 0), (7, 15), (8, 16), (31, 31), (13, 30)):
        xi = x.clone()
        xi[1, r, c, 1] = float("inf")
        block.cache(xi, out)
        near = torch.zeros((2, 32, 32), dtype=torch.bool, device="cuda")
        near[1, max(0, r - 1):r + 2, max(0, c - 1):c + 2] = True
        assert torch.equal(out[~near], ref[~near])
        assert not bool(torch.isfinite(out[near].float()).all())


@pytest.mark.parametrize("shift", [0, 1024])
def test_output_over_the_images(shift):
    import torch
    nf, L, p, x = _layer(3, 32, 32, 9)
    want, ys = _reference(x, p)
    buf = torch.zeros(shift + 3 * 32 * 32 * 64, dtype=torch.bfloat16, device="cuda")
    buf[:x.numel()] = x.flatten()
    _cache(nf, nf.Block([L]), buf[:x.numel()], buf[shift:], 4)
    _check(buf[shift:].view(3, 32, 32, 64), want, ys)
