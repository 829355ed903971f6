"""GPU: emc_update by the rows' pairs at the edges of what finds a row tile to be over: the
look at eight of its rows in 256 frames (more than 256 of 2048 non-zero) and a block of 128
rows x 256 frames (512 pairs), with every row and tile total below its own limit or far above.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16_split", "fp16_split"])
def test_update_around_the_blocks(precision):
    """A row tile each: empty; dense; 512 and 513 pairs in one block (4 or 5 a row); the looked-at
    block with 256 and 257 of its 2048 elements non-zero (8 rows, 32 or 33 pairs). The sums
    have at most 2 n + 1 exact products (hi and lo planes) of one sign, each addition off by at
    most 2^-23 of its result: 2 (n + 1) 2^-23 of the sum."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 16)
    quat, w = emc.quat_generate(4)
    n_rot, n_pix, n_data = quat.shape[0], det.q.shape[0], 5300
    ctx = emc.Context(16, det.q, quat, w, n_data, precision=precision)
    rng = np.random.default_rng(5)
    K = rng.poisson(0.7, size=(n_data, n_pix)).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    b = ctx.buffer_sizes(n_rot)
    P = np.zeros((b.rows, ctx.ld_data), dtype=np.float32)
    mid = ctx.ld_data // 512 * 256  # the looked-at frames
    for t in range(n_rot // 128):
        rows = 128 * t + np.arange(128)
        kind = t % 6
        if kind == 1:
            P[rows, :n_data] = 0.01 + rng.random((128, n_data))
        elif kind in (2, 3):
            for r in rows:
                P[r, 512 + rng.permutation(256)[:4]] = 0.01 + rng.random(4)
            if kind == 3:
                P[rows[7], 512:768] = 0.0
                P[rows[7], 512 + rng.permutation(256)[:5]] = 0.5
        elif kind in (4, 5):
            for r in rows[::16]:
                P[r, mid + rng.permutation(256)[:32]] = 0.01 + rng.random(32)
            if kind == 5:
                at = np.nonzero(P[rows[16], mid:mid + 256] == 0)[0][0]
                P[rows[16], mid + at] = 0.5
    scale, dt = (2.0 ** 14, torch.float16) if precision == "fp16_split" else (1.0, torch.bfloat16)
    x = torch.as_tensor(P, device="cuda") * scale
    hi = x.to(dt)
    lo = (x - hi.float()).to(dt)
    planes = torch.stack([hi, lo]).contiguous()
    held = ((hi.double() + lo.double()) / scale)[:n_rot, :n_data]
    Num, den = ctx.update(planes.view(torch.uint8).reshape(-1), n_rot)
    want = held @ torch.as_tensor(K, device="cuda").double()
    n = (held != 0).sum(1, keepdim=True).double()
    tol = 2.0 * (n + 1) * 2.0 ** -23
    assert bool(((Num[:n_rot, :n_pix].double() - want).abs() <= tol * want).all())
    wden = held.sum(1)
    assert bool(((den[:n_rot].double() - wden).abs() <= tol[:, 0] * wden).all())
    assert ctx.status() == 0
