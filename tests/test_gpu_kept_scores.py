"""GPU: pass 2 of a bound-pruned iteration without stored scores, from the scores
pass 1 kept of its live tiles, against the dense two-pass form from the same models.
The kept scores live in the last L's buffer (6 B a rotation and pixel against 4.1 B a
rotation and frame), so few pixels and many frames leave only some tiles a place
(the others are contracted again), few frames all of them. The model's bar is the
pruned iterations' (FP32 rounding of the M-step's order): 1e-6 relative L2.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("model,precision", [("poisson", "bf16_split"), ("poisson", "fp16_split"),
                                             ("poisson_fluence", "bf16_split")])
@pytest.mark.parametrize("n_data,chunk", [(100, 0), (3000, 0), (3000, 384)])
def test_kept_scores_equal_recomputed(model, precision, n_data, chunk):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    ds = synth.make_dataset(16, 16, n_data, 1.0, radius=4.0,
                            fluence_sigma=0.2 if model == "poisson_fluence" else 0.0)
    quat, w = emc.quat_generate(3)
    floor = 1e-10 * float(ds.model_start.mean())
    kw = dict(precision=precision, model=model, w_floor=floor, rot_chunk=chunk)
    a = emc.Context(16, ds.q, quat, w, n_data, **kw)
    d = emc.Context(16, ds.q, quat, w, n_data, dense_estep=True, **kw)
    K = torch.as_tensor(ds.K, device="cuda")
    a.set_frames(K)
    d.set_frames(K)
    g = torch.as_tensor(ds.model_start.astype(np.float32), device="cuda")
    planes = 3 if precision == "bf16_split" else 2
    room = 2 * planes * a.sizes_all.rows * a.ld_pix // (4 * 33792)  # tiles whose scores fit
    for it in range(4):
        out, st = a.iteration(g)
        ref, _ = d.iteration(g)
        assert st["device_status"] == 0
        if it:
            assert st["pass1_pruned"] == 1
            # both sides of the rule are met: every live tile kept (100 frames, three planes), or
            # only some
            assert (st["pass1_exact"] <= room) == (n_data == 100 and planes == 3)
        assert _rel(out, ref) <= 1e-6
        lse, want = a.iteration_lse(), d.iteration_lse()
        assert float((lse - want).abs().max()) <= 1e-4
        g = ref
