"""GPU: the FP32 update over responsibilities with whole frames of exact zeros,
against the sum in FP64. Frame counts around the 4096 taken at a time; row tiles
with no, one, few and every frame non-zero. A row's sum of n non-negative products
is formed in order with one rounding each: |error| <= n 2^-24 of the sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_data", [1, 300, 4096, 4200])
def test_update_skips_zero_frames_exactly(n_data):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(14, 16)
    quat, w = emc.quat_generate(2)
    n_rot, n_pix = quat.shape[0], det.q.shape[0]
    ctx = emc.Context(16, det.q, quat, w, n_data, precision="fp32")
    rng = np.random.default_rng(n_data)
    K = rng.poisson(0.7, size=(n_data, n_pix)).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    b = ctx.buffer_sizes(n_rot)
    P = np.zeros((b.rows, b.ld_data), dtype=np.float32)
    for t, share in enumerate([0.0, 1.0, 0.02, 0.5, None, 0.001, 0.2] * 3):
        r = slice(64 * t, min(64 * t + 64, n_rot))
        if r.start >= n_rot:
            break
        if share is None:
            P[r.start + 3, n_data - 1] = 0.25  # one pair of the tile
        else:
            P[r, :n_data] = rng.random((r.stop - r.start, n_data)) * (rng.random(n_data) < share)
    buf = torch.as_tensor(P, device="cuda").view(torch.uint8).reshape(-1)
    Num, den = ctx.update(buf, n_rot)
    num = Num[:n_rot, :n_pix].double().cpu().numpy()
    want = P[:n_rot, :n_data].astype(np.float64) @ K
    cnt = (P[:n_rot] != 0).sum(1)
    tol = (cnt + 1)[:, None] * 2.0 ** -24
    assert np.all(np.abs(num - want) <= tol * want)
    wden = P[:n_rot].astype(np.float64).sum(1)
    assert np.all(np.abs(den[:n_rot].double().cpu().numpy() - wden) <= tol[:, 0] * wden)
