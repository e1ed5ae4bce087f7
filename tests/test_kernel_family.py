"""nf_layer_kernel_family names what a step runs, and the benchmark's byte counts follow it (host only)."""
import ctypes as C

import bench
from paper_2402_14139_b200 import build, nf


def _families(Cin, Cout, H, W, F, N):
    L = nf.lib()
    h = L.nf_layer_create(Cin, Cout, H, W, F, 10)
    o = nf.nf_layer_opts(N, 1, 0, nf.NF_BF16, 0.9, 1e-5, 0.1, 0, 0, 0)
    assert L.nf_layer_configure(h, C.byref(o)) == nf.NF_OK
    fam = [L.nf_layer_kernel_family(h, k).decode() for k in range(10)]
    L.nf_layer_destroy(h)
    return fam


def test_weight_and_input_gradient_are_named_apart():
    build.build()
    small = _families(64, 64, 14, 14, 16, 10)      # a map that no tile divides, below 8192 pixels: only the weight gradients
    assert [small[k] for k in (0, 1, 2, 3, 7)] == ["cuda-core", "tcgen05", "cuda-core", "tcgen05", "cuda-core"]
    large = _families(64, 64, 14, 14, 16, 60)
    assert [large[k] for k in (0, 1, 2, 3, 7)] == ["tcgen05"] * 5 and large[9] == ""


def test_gradient_at_h_is_counted_where_it_is_written():
    l, N = dict(Cin=64, Cout=64, H=16, W=16, F=16, stride=1, pool=False), 8
    fam = ["tcgen05"] * 4 + ["separate", "stored", "stored", "cuda-core"]
    apart, together = bench.op_model(l, N, 10, 2, fam + ["separate"]), bench.op_model(l, N, 10, 2, fam + ["head"])
    h = 2 * N * 16 * 16 * 16
    assert apart["aux_wgrad"][2] - together["aux_wgrad"][2] == 2 * h and together["head"][2] - apart["head"][2] == h
    assert apart["aux_dgrad"][0] == "alu" and apart["aux_wgrad"][0] == "tensor"
