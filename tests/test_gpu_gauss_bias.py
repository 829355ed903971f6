"""GPU: the Gaussian bias log w_j - sum_i W_ij^2 / (2 sigma^2) against FP64 sums of the W that
the planes of L hold (s W = hi + mid + lo, s a power of two), on the tile kernels and on
the one-launch form. The planes hold s W to 2^-25 (half of FP16's smallest step) where
they are not exact, so each square is off by 2 W 2^-25 / s; the sums add no rounding of
their own above 2^-44 (W^2 rounded to FP32 before it is summed would add 2^-25 a term).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_quat", [1, 6])
def test_bias_is_the_sum_of_squares(n_quat):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 64)
    quat, w = emc.quat_generate(n_quat)
    n, n_pix = quat.shape[0], det.q.shape[0]
    ctx = emc.Context(64, det.q, quat, w, 4, model="gaussian", sigma=0.7)
    K = torch.zeros(4, n_pix, dtype=torch.int32, device="cuda")
    K[:, 0] = 1  # few photons: a large s
    ctx.set_frames(K)
    g = torch.Generator(device="cuda").manual_seed(1)
    grid = 1.0 + torch.rand(64, 64, 64, generator=g, device="cuda")
    L, bias = ctx.expand(grid, 0, n)
    rows = ctx.sizes_all.rows
    sW = L.view(torch.float16).view(3, rows, ctx.ld_pix).double().sum(0)[:n, :n_pix]
    top = float(sW.max())
    s = 2.0 ** np.round(np.log2(top / 1.9))  # W of the interpolated model: at most 2, near it
    W = sW / s
    assert 1.0 <= float(W.min()) and 1.5 < float(W.max()) <= 2.0 and s >= 64
    sq = (W * W).sum(1)
    want = torch.as_tensor(np.log(w), device="cuda") - sq / (2 * 0.7 ** 2)
    tol = (2 * W.sum(1) * 2.0 ** -25 / s + sq * 2.0 ** -44) / (2 * 0.7 ** 2) + 1e-12
    assert bool(((bias[:n] - want).abs() <= tol).all())
    assert ctx.status() == 0
