"""GPU: the sparse E-step from the frames' non-zero lists, which scores only the
candidate pairs that can matter, against the same step from the frames' rows, which
scores them all. Both use the same split of log W: S to FP32 rounding of the small
part (|rest| N_k 2^-24 sqrt(n) < 1e-4 here), so lse within 1e-4 and P within 2e-4
of the larger; a pair that one form leaves out has P = 0 in the other.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16_split", "fp16_split", "fp32"])
@pytest.mark.parametrize("photons", [0.02, 3.0])
def test_choice_changes_nothing(precision, photons):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    ds = synth.make_dataset(32, 32, 130, photons, radius=8.0)
    np.minimum(ds.K, 256, out=ds.K)  # the largest count the 16-bit frames hold
    ds.K[7] = 0  # an empty frame
    quat, w = emc.quat_generate(3)
    n_rot, M = quat.shape[0], 200
    rng = np.random.default_rng(3)
    cand = np.argsort(rng.random((130, n_rot)), axis=1)[:, :M].astype(np.int32)
    grid = torch.as_tensor(ds.model_start.astype(np.float32), device="cuda")
    got = []
    for lists in (True, False):
        ctx = emc.Context(32, ds.q, quat, w, 130, precision=precision, n_cand=M, sparse_k=lists,
                          w_floor=1e-10 * float(ds.model_start.mean()))
        ctx.set_frames(torch.as_tensor(ds.K, device="cuda"))
        ctx.set_candidates(torch.as_tensor(cand, device="cuda"))
        L, bias = ctx.expand(grid, 0, n_rot)
        P, lse = ctx.sparse_estep(L, bias)
        assert ctx.status() == 0
        got.append((P[:130].double(), lse[:130]))
    (Pa, la), (Pb, lb) = got
    assert float((la - lb).abs().max()) <= 1e-4
    assert bool(((Pa - Pb).abs() <= 2e-4 * torch.maximum(Pa, Pb) + 1e-44).all())
