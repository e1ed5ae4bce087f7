"""fp32 BatchNorm backward where the mean is large against the standard deviation: dy = gamma*invstd * (dz - sum(dz)/M - xhat *
sum(dz*xhat)/M) has to be formed from y - mu.  Written as s*dz + k1*y + k0 it adds two terms of the size of
s * sum(dz*xhat)/M * |mu|/sigma that cancel, and loses that ratio in accuracy."""
import numpy as np
import pytest

from paper_2402_14139_b200 import synth

pytestmark = pytest.mark.gpu

# A term of dy passes through at most ten roundings of 2^-24 (difference, invstd, product, coefficient, 1/M, two products, two sums,
# scale); the variance that is read back was rounded once more and divided: 12 units of the largest sum of the terms' sizes.  The
# other form is off by |mu|/sigma units of sum(dz*xhat)/M, here more than a hundred.
UNITS = 12 * 2.0 ** -24


def _bound(scale, dz, m1, xh, m2):
    return UNITS * (scale * (np.abs(dz) + np.abs(m1) + np.abs(xh * m2))).max()


def test_layer_dy_with_a_large_mean():
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    N, C, S = 2, 16, 24
    L = nf.Layer(C, C, S, S, 8, 10, N, dtype=nf.NF_F32, bn_momentum=1.0)   # the running statistics become the batch's
    W = np.zeros((C, C, 3, 3), dtype=np.float32)
    W[:, :, 1, 1] = 0.5 + synth.uniform01(5, 1, C * C).reshape(C, C)       # centre tap only: no effect of the padding on the mean
    L.set_param("W", W)
    # the gradient at the activation is the same everywhere but at the edge (positive filters, every h positive, equal quadrants, one
    # label), so that sum(dz*xhat) is as large as it can be
    L.set_param("Wa", (0.1 * synth.uniform01(5, 2, 8 * C * 9)).astype(np.float32).reshape(8, C, 3, 3))
    L.set_param("ba", np.ones(8, dtype=np.float32))
    L.set_param("Wf", np.repeat(0.2 * synth.normal(5, 3, (10, 8)), 4, axis=1).astype(np.float32))
    x = torch.from_numpy((100.0 + synth.normal(5, 4, (N, S, S, C))).astype(np.float32)).cuda()
    L.step(x, torch.full((N,), 3, dtype=torch.int32, device="cuda"), 0.0, torch.zeros(1, device="cuda"), L.new_act())
    torch.cuda.synchronize()
    assert L.status() == 0
    f64 = lambda t: t.double().cpu().numpy()
    M = N * S * S
    Y, da, dy = f64(L.stored("y")), f64(L.stored("da")), f64(L.stored("dy"))
    mu, var = L.get_param("rmean").astype(np.float64), L.get_param("rvar").astype(np.float64) * (M - 1) / M
    invstd = 1.0 / np.sqrt(var + 1e-5)
    m1, m2 = (L.get_param(k, nf.NF_K_GRAD).astype(np.float64) / M for k in ("beta", "gamma"))
    xh = (Y - mu) * invstd
    assert np.abs(mu * invstd).min() > 300 and np.abs(m2).max() > 0.3 * np.abs(da).max()
    dz = np.where(xh > 0, da, 0.0)
    want = invstd * (dz - m1 - xh * m2)
    sure = np.abs(xh) > 1e-2                                               # the mask of the others hangs on the rounding of shift
    assert sure.mean() > 0.9
    assert np.abs(dy - want)[sure].max() <= _bound(invstd, dz, m1, xh, m2)
    L.close()


def test_projection_dy_with_a_large_mean():
    """The gradient at the projection's conv output is not exposed; input channels that are 1 at one pixel, 0 elsewhere and have zero
    weight bring its value at that pixel out as their weight gradient."""
    import torch
    from paper_2402_14139_b200 import nf
    nf.lib()
    nf.nf_set_stream(None)
    N, Cin, Cout, S = 2, 64, 32, 8                                          # 8 x 8 outputs of a 16 x 16 map
    GP = nf.Projection(Cin, Cout, 2 * S, 2 * S, N, dtype=nf.NF_F32, bn_momentum=1.0)
    W = np.zeros((Cout, Cin), dtype=np.float32)
    W[:, 0] = 0.5 + synth.uniform01(6, 1, Cout)
    GP.set_param("W", W)
    xb = np.zeros((N, 2 * S, 2 * S, Cin), dtype=np.float32)
    xb[..., 0] = 300.0 + synth.normal(6, 2, (N, 2 * S, 2 * S))
    at = [(k % N, (k // N) // S, (k // N) % S) for k in range(1, Cin)]       # the output pixel channel k looks at
    for k, (n, i, j) in enumerate(at, 1):
        xb[n, 2 * i, 2 * j, k] = 1.0
    dz = (1.0 + 0.5 * synth.normal(6, 3, (N, S, S, Cout))).astype(np.float32)
    xd = torch.from_numpy(xb).cuda()
    s = GP.new_out()
    GP.forward(xd, s)
    Y = xb[:, ::2, ::2, 0].astype(np.float32)[..., None] * W[:, 0]           # one product per output: exactly the stored conv output
    mu = GP.get_param("rmean").astype(np.float64)
    M = N * S * S
    invstd = 1.0 / np.sqrt(GP.get_param("rvar").astype(np.float64) * (M - 1) / M + 1e-5)
    dz += (0.5 * ((Y - mu) * invstd)).astype(np.float32)                     # a gradient that goes along with xhat: a large sum(dz*xhat)
    GP.backward(xd, torch.from_numpy(dz).cuda(), 0.0)
    torch.cuda.synchronize()
    m1, m2 = (GP.get_param(k, nf.NF_K_GRAD).astype(np.float64) / M for k in ("beta", "gamma"))
    gW = GP.get_param("W", nf.NF_K_GRAD).astype(np.float64)
    xh = (Y.astype(np.float64) - mu) * invstd
    assert np.abs(mu * invstd).min() > 200 and np.abs(m2).min() > 0.2
    want = invstd * (dz - m1 - xh * m2)
    bound = _bound(invstd, dz, m1, xh, m2)
    for k, (n, i, j) in enumerate(at, 1):
        assert np.abs(gW[:, k] - want[n, i, j]).max() <= bound, k
    GP.close()
