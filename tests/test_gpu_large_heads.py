"""The linear head at the boundaries of its forms: the tiled products of large batches (tiles of 64 and of 32 rows, remainders in every
extent, class counts that no 16-byte load divides), the sizes on both sides of their threshold, and maps of one pixel, whose head is
the one-block-per-sample kernel with the batch sums after it.  fp32 layers on tiny maps, so that the tolerance is 1e-4."""
import pytest

from tests import parity_util as pu

pytestmark = pytest.mark.gpu


def _c(N, F, K, S=2, C=16):
    return dict(N=N, Cin=C, Cout=C, H=S, W=S, F=F, classes=K, stride=1, pool=False)


CASES = [
    _c(8605, 64, 201),          # 540 tiles of 64 x 64: logits and input gradient on tiles of 64 rows, K % 4 = 1
    _c(7013, 72, 260),          # tiles of 64 rows with whole 16-byte loads, inputs 4 * 72 = 288 = 4.5 tiles
    _c(3301, 24, 67),           # tiles of 32 rows
    _c(1023, 16, 256),          # 2^24 - 2^14 multiply-adds: below the threshold
    _c(1024, 16, 256),          # 2^24: the first of the tiled products
    _c(203, 8, 10, S=1),        # one pixel: batch sums of 50 groups of four and three more
    _c(3, 8, 10, S=1),          # fewer samples than chains
    _c(261, 24, 33, S=1),
]


@pytest.mark.parametrize("ci", range(len(CASES)))
def test_fp32_step_with_a_head_at_a_boundary(ci):
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    pu.check_step(nf, torch, CASES[ci], seed=1300 + ci, dtype=nf.NF_F32, lr=0.02, steps=1)
