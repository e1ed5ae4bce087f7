"""Edges of the tiles and of the dispatch rules: the weight gradient with 128 output channels on the M side, first layers over 16
padded channels, the CUDA-core convolutions and the per-sample heads (the large-batch ones: test_gpu_large_heads.py).  Tolerances are those of parity_util.TOL."""
import pytest

from tests import parity_util as pu

pytestmark = pytest.mark.gpu

BF16 = [
    # weight gradient, 128 output channels per CTA: one or two chunks of input channels
    dict(N=37, Cin=64, Cout=128, H=16, W=16, F=16, classes=10, stride=1, pool=False),   # one image per tile, one chunk
    dict(N=33, Cin=128, Cout=128, H=16, W=16, F=16, classes=10, stride=1, pool=False),  # two chunks
    dict(N=35, Cin=192, Cout=256, H=8, W=8, F=16, classes=10, stride=1, pool=False),    # two images per tile, an odd number of them
    dict(N=9, Cin=128, Cout=128, H=4, W=4, F=8, classes=10, stride=1, pool=False),      # eight images per tile, the last tile nearly empty
    dict(N=3, Cin=64, Cout=128, H=24, W=32, F=16, classes=10, stride=1, pool=True),
    dict(N=42, Cin=128, Cout=128, H=14, W=14, F=16, classes=10, stride=1, pool=False),  # tiles over the right and lower edge
    dict(N=3, Cin=128, Cout=128, H=4, W=8, F=8, classes=10, stride=1, pool=False),      # fewer pixels than one tile
    # first layers: 3 and 4 channels, widths the 14-column groups divide and do not divide
    dict(N=3, Cin=3, Cout=64, H=28, W=28, F=8, classes=10, stride=1, pool=False),
    dict(N=9, Cin=4, Cout=64, H=32, W=32, F=16, classes=10, stride=1, pool=True),
    dict(N=2, Cin=3, Cout=64, H=64, W=128, F=16, classes=10, stride=1, pool=False),
    # per-sample heads: few classes, many, one sample
    dict(N=63, Cin=64, Cout=64, H=8, W=8, F=12, classes=3, stride=1, pool=False),
    dict(N=130, Cin=64, Cout=64, H=8, W=8, F=40, classes=101, stride=1, pool=False),
    dict(N=1, Cin=64, Cout=64, H=8, W=16, F=8, classes=10, stride=1, pool=False),
]

FP32 = [
    dict(N=1, Cin=3, Cout=16, H=5, W=7, F=4, classes=10, stride=1, pool=False),      # less than one tile of pixels
    dict(N=2, Cin=17, Cout=33, H=9, W=15, F=6, classes=3, stride=1, pool=False),     # no extent a multiple of four
    dict(N=3, Cin=24, Cout=65, H=8, W=8, F=10, classes=10, stride=2, pool=False),    # one channel over a 64-wide tile
    dict(N=30, Cin=20, Cout=128, H=18, W=18, F=16, classes=10, stride=1, pool=True),  # tiles of 64 x 64 with a remainder
    dict(N=5, Cin=32, Cout=32, H=33, W=5, F=32, classes=100, stride=1, pool=False),
]


@pytest.mark.parametrize("ci", range(len(BF16)))
def test_bf16_step_at_tile_edges(ci):
    import torch
    from paper_2402_14139_b200 import nf
    pu.check_step(nf, torch, BF16[ci], seed=900 + ci, dtype=nf.NF_BF16, lr=0.02, steps=2)


@pytest.mark.parametrize("ci", range(len(FP32)))
def test_fp32_step_at_tile_edges(ci):
    import torch
    from paper_2402_14139_b200 import nf
    pu.check_step(nf, torch, FP32[ci], seed=950 + ci, dtype=nf.NF_F32, lr=0.02, steps=2)
