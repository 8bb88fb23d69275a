"""Cost-model kernels at the edges of their sample tiles (64 forward; 32 to 80
backward), around the batch that first has room for a copy of the gradient in
its scratch, and with every buffer off a 16-byte boundary.

Tolerances: an output is a sum of at most n fp32 terms whose rounding errors
stay below n * 2^-24 of the sum of the terms' magnitudes; n is 64 + F for the
forward pass, and the gradients' sums over the batch run through chains of at
most 16 samples, the tiles of one CTA and the CTAs of one copy (below 400 in
all), so 1e-4 of the largest magnitude leaves a factor of four."""
import ctypes

import numpy as np
import pytest

from oracle import mlp_ref
from paper_1709_00700_gb300 import pv
from tests.test_gpu_mlp import H, _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,F", [(31, 45), (32, 45), (33, 45), (55, 45), (56, 45), (65, 64), (66, 64), (79, 20), (81, 20),
                                 (4865, 3), (9729, 60), (24_321, 17)])
@pytest.mark.parametrize("shift", [0, 1])
def test_tiles(B, F, shift):
    import torch
    ctx = pv.Context(0)
    X, t, mu, sigma, p = _case(B, F, B + F)

    def dev(a):
        buf = torch.zeros(np.size(a) + shift, dtype=torch.float32, device="cuda")
        buf[shift:] = torch.tensor(np.ravel(a), dtype=torch.float32, device="cuda")
        return buf

    def ptr(b):
        return ctypes.c_void_p(b.data_ptr() + 4 * shift)

    dp, dX, dmu, dsig, dt = dev(p), dev(X), dev(mu), dev(sigma), dev(t)
    y, act, dz = dev(np.zeros(B)), dev(np.zeros(B * 2 * H)), dev(np.full(B * (2 * H + 1), np.nan))
    grad, loss = dev(np.full(len(p), 7.0)), dev(np.zeros(1))
    torch.cuda.synchronize()
    lib = ctx.lib
    for _ in range(2):  # the scratch holds the first call's sums
        assert lib.pv_mlp_forward(ctx.h, ptr(dp), ptr(dX), ptr(dmu), ptr(dsig), B, F, ptr(y), ptr(act)) == 0
        assert lib.pv_mlp_backward(ctx.h, ptr(dp), ptr(dX), ptr(dmu), ptr(dsig), ptr(act), ptr(y), ptr(dt), B, F,
                                   ptr(dz), ptr(grad), ptr(loss)) == 0
    ctx.stream.synchronize()
    r = lambda a: np.asarray(a, np.float32).astype(np.float64)  # noqa: E731
    yr, cache = mlp_ref.forward(r(p), r(X), r(mu), r(sigma), H)
    gr = mlp_ref.backward(r(p), cache, yr, r(t), H)
    assert np.abs(y[shift:].cpu().numpy() - yr).max() <= 1e-4 * np.abs(yr).max()
    assert np.abs(grad[shift:].cpu().numpy() - gr).max() <= 1e-4 * np.abs(gr).max()
    assert abs(loss[shift:].item() - mlp_ref.loss(yr, r(t))) <= 1e-4 * mlp_ref.loss(yr, r(t))
    ctx.close()
