"""GPU: the sparse update over rows whose lists hold no, few and many non-zero
weights (Eq. 2.11 over candidate sets), against the sum written out in FP64.

Every rotation is a candidate of every frame, so a row's list has n_data = 1500
pairs (more than the 1024 the kernel packs at a time); the weights P are set to
zero except for the first `keep[j]` frames of row j's random order. Num_ij is an
FP32 sum of at most keep[j] non-negative products, each rounded once and added
once: |error| <= 2 keep 2^-24 of the sum, and the same for den_j.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lists", [True, False])
@pytest.mark.parametrize("n_data", [7, 1024, 1500])
def test_update_over_nonzero_weights(lists, n_data):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(14, 16)
    quat, w = emc.quat_generate(1)
    n_rot, n_pix = quat.shape[0], det.q.shape[0]
    ctx = emc.Context(16, det.q, quat, w, n_data, n_cand=n_rot, sparse_k=lists)
    rng = np.random.default_rng(31)
    K = rng.poisson(0.7, size=(n_data, n_pix)).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    cand = np.argsort(rng.random((n_data, n_rot)), axis=1).astype(np.int32)
    ctx.set_candidates(torch.as_tensor(cand, device="cuda"))
    keep = np.minimum(rng.choice([0, 1, 2, 3, 5, 8, 100, 1500], size=n_rot), n_data)
    P = np.zeros((n_rot, n_data), dtype=np.float32)
    for j in range(n_rot):
        k = rng.permutation(n_data)[:keep[j]]
        P[j, k] = rng.random(len(k)).astype(np.float32)
    slots = np.zeros((ctx.ld_data, n_rot), dtype=np.float32)
    slots[:n_data] = np.take_along_axis(P.T, cand.astype(np.int64), axis=1)
    Num, den = ctx.sparse_update(torch.as_tensor(slots, device="cuda"))
    num = Num[:n_rot, :n_pix].double().cpu().numpy()
    want = P.astype(np.float64) @ K
    tol = 2.0 * (keep[:, None] + 1) * 2.0 ** -24
    assert np.all(np.abs(num - want) <= tol * want)
    wden = P.astype(np.float64).sum(1)
    assert np.all(np.abs(den[:n_rot].double().cpu().numpy() - wden) <= tol[:, 0] * wden)
    assert ctx.status() == 0
