"""GPU: the bound that chooses candidate pairs in the sparse E-step (frames as lists) when
the bias is far larger than FP32 resolves: a model scaled far above the counts.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", [0.0, 1.5e9, 3e12])
@pytest.mark.parametrize("precision", ["bf16_split", "fp16_split", "fp32"])
def test_large_bias_drops_no_pair(precision, base):
    """L = 0, so S_jk = bias_j = -(base + 40 + 1.25 j) whatever the frame: P_jm = (1 - e^-1.25)
    e^(-1.25 m) over 64 candidates, all above FP32's zero. S - lse is off by one FP64 rounding
    of 3e12 (2.5e-4) twice, the exponential of at most 80 by 80 x 2^-23 in its argument and
    2^-21 itself: 6e-4 relative (2e-5 below 1e10)."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(14, 16)
    quat, w = emc.quat_generate(2)
    n_pix, n_data, M = det.q.shape[0], 5, 64
    ctx = emc.Context(16, det.q, quat, w, n_data, precision=precision, n_cand=M, sparse_k=True)
    K = np.zeros((n_data, n_pix), dtype=np.int32)
    K[:, :8] = 1
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    cand = torch.arange(M, dtype=torch.int32, device="cuda").repeat(n_data, 1).contiguous()
    ctx.set_candidates(cand)
    b = ctx.sizes_all
    L = torch.zeros(b.logw_bytes, dtype=torch.uint8, device="cuda")
    bias = -(base + 40 + 1.25 * torch.arange(b.rows, dtype=torch.float64, device="cuda"))
    P, lse = ctx.sparse_estep(L, bias)
    want = -np.expm1(-1.25) * np.exp(-1.25 * np.arange(M))
    got = P[:n_data].double().cpu().numpy()
    assert np.all(np.abs(got / want - 1) <= (6e-4 if base > 1e10 else 2e-5))
    assert ctx.status() == 0


def test_infinite_bias_is_scored():
    """A bias of -infinity is no candidate's best; one of NaN is met and reported."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(14, 16)
    quat, w = emc.quat_generate(2)
    ctx = emc.Context(16, det.q, quat, w, 2, n_cand=3, sparse_k=True)
    ctx.set_frames(torch.ones(2, det.q.shape[0], dtype=torch.int32, device="cuda"))
    ctx.set_candidates(torch.tensor([[0, 1, 2], [3, 4, 5]], dtype=torch.int32, device="cuda"))
    b = ctx.sizes_all
    L = torch.zeros(b.logw_bytes, dtype=torch.uint8, device="cuda")
    bias = torch.zeros(b.rows, dtype=torch.float64, device="cuda")
    bias[1] = -torch.inf
    P, lse = ctx.sparse_estep(L, bias)
    assert ctx.status() == 0
    assert torch.allclose(P[0], torch.tensor([0.5, 0.0, 0.5], device="cuda"), rtol=1e-6)
    bias[4] = torch.nan
    ctx.sparse_estep(L, bias)
    assert ctx.status() == -6
