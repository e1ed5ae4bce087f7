"""Tensor-core kernels on map sizes that no 128-pixel tile divides (7, 14, 28, odd sizes): tiles that hang over the right and
lower edge and over the last image, for every role a kernel has in a step.  Tolerances are those of parity_util.TOL."""
import pytest

from tests import parity_util as pu

pytestmark = pytest.mark.gpu

# the tensor cores take such maps from 8192 output pixels on
CASES = [
    dict(N=168, Cin=64, Cout=64, H=7, W=7, F=16, classes=10, stride=1, pool=False),    # one pixel of many images per tile, images missing
    dict(N=42, Cin=64, Cout=256, H=14, W=14, F=16, classes=10, stride=1, pool=False),  # 2 x 2 patches, 256-wide channel tile
    dict(N=235, Cin=64, Cout=128, H=13, W=9, F=16, classes=10, stride=2, pool=False),  # odd input, stride 2
    dict(N=11, Cin=64, Cout=128, H=28, W=28, F=32, classes=10, stride=1, pool=False),
    dict(N=13, Cin=64, Cout=64, H=20, W=36, F=24, classes=10, stride=1, pool=False),   # a width the folded kernels take, a height they do not
    dict(N=550, Cin=64, Cout=64, H=6, W=10, F=8, classes=10, stride=1, pool=True),     # pool: the aux network sees 3 x 5
    dict(N=102, Cin=3, Cout=64, H=9, W=9, F=8, classes=10, stride=1, pool=False),      # zero-padded input channels
    dict(N=330, Cin=64, Cout=64, H=5, W=5, F=128, classes=10, stride=1, pool=False),   # wide auxiliary network
    dict(N=15, Cin=64, Cout=64, H=17, W=33, F=16, classes=10, stride=1, pool=False),
]


@pytest.mark.parametrize("ci", range(len(CASES)))
def test_step_on_maps_no_tile_divides(ci):
    import torch
    from paper_2402_14139_b200 import nf
    c = CASES[ci]
    P, _, _ = pu.seeded_case(c, 1, bf16=True)
    G = pu.gpu_layer(nf, c, P, nf.NF_BF16)
    assert [G.kernel_family(k) for k in range(4)] == ["tcgen05"] * 4
    G.close()
    pu.check_step(nf, torch, c, seed=700 + ci, dtype=nf.NF_BF16, lr=0.02, steps=2)
