"""GPU: emc_update where the caller's P holds numbers in its padding frames. They carry no
counts, so Num and den are those of a P with zeros there, on every path: the rows' pairs,
the planes, FP32.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n_data", [("bf16_split", 5301), ("fp16_split", 5301),
                                              ("bf16_split", 301), ("bf16", 301), ("fp32", 301)])
def test_padding_frames_add_nothing(precision, n_data):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 16)
    quat, w = emc.quat_generate(4 if n_data > 1000 else 2)
    n_rot = quat.shape[0]
    ctx = emc.Context(16, det.q, quat, w, n_data, precision=precision)
    K = np.random.default_rng(3).poisson(0.7, size=(n_data, det.q.shape[0])).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    b = ctx.buffer_sizes(n_rot)
    g = torch.Generator(device="cuda").manual_seed(n_data)
    x = torch.zeros((b.rows, ctx.ld_data), device="cuda")
    rows = torch.arange(n_rot, device="cuda")
    for _ in range(3):
        x[rows, torch.randint(n_data, (n_rot,), generator=g, device="cuda")] = 0.5
    y = x.clone()
    y[:n_rot:3, n_data:n_data + 2] = 0.75
    y[1, n_data:] = 0.25

    def update(p):
        if precision != "fp32":
            dt = torch.float16 if precision == "fp16_split" else torch.bfloat16
            p = p * (2.0 ** 14 if precision == "fp16_split" else 1.0)
            p = torch.stack([p.to(dt), torch.zeros_like(p).to(dt)])
        return ctx.update(p.contiguous().view(torch.uint8).reshape(-1), n_rot)

    (Na, da), (Nb, db) = update(x), update(y)
    assert torch.equal(Na[:n_rot], Nb[:n_rot]) and torch.equal(da[:n_rot], db[:n_rot])
    assert ctx.status() == 0
