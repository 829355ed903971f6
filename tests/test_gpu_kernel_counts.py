"""GPU: emc_iter_stats.kernels is the number of kernels that a call launches: a context's
k-th call with stats, against the kernel nodes of another context's k-th call, captured.
"""
import functools

import numpy as np
import pytest

from test_gpu_capture import capture, rt  # noqa: F401

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=None)
def dataset(N, D, n_data, photons, fluence):
    from paper_1409_4256_gb300 import synth
    return synth.make_dataset(N, D, n_data, photons, radius=4.0, fluence_sigma=fluence)


def contexts(N, D, n_quat, n_data, photons, **kw):
    import torch
    from paper_1409_4256_gb300 import emc
    ds = dataset(N, D, n_data, photons, 0.2 if kw.get("model", "poisson") != "poisson" else 0.0)
    quat, w = emc.quat_generate(n_quat)
    kw.setdefault("w_floor", 1e-10 * float(ds.model_start.mean()))
    K = torch.as_tensor(np.minimum(ds.K, 250), device="cuda")
    out = []
    for _ in range(2):
        ctx = emc.Context(N, ds.q, quat, w, n_data, **kw)
        ctx.set_frames(K)
        out.append(ctx)
    return out, torch.as_tensor(ds.model_start.astype(np.float32), device="cuda"), ds


@pytest.mark.parametrize("kw", [
    dict(), dict(store_scores=True), dict(dense_estep=True), dict(rot_chunk=640),
    dict(rot_chunk=640, store_scores=True), dict(precision="fp16_split"),
    dict(precision="bf16"), dict(precision="bf16", store_scores=True), dict(precision="fp32"),
    dict(precision="fp32", store_scores=True), dict(model="poisson_fluence"),
    dict(model="poisson_fluence", store_scores=True, rot_chunk=640),
    dict(model="poisson_fluence", dense_estep=True),
    dict(model="gaussian", precision="fp16_split", sigma=3.0),
    dict(model="gaussian", precision="fp16_split", sigma=3.0, rot_chunk=640)])
@pytest.mark.parametrize("size", [(16, 14, 3, 300, 0.5), (16, 60, 4, 5303, 0.15)])
def test_iterations(rt, kw, size):  # noqa: F811
    import torch
    (a, b), grid, _ = contexts(*size, **kw)
    stream = torch.cuda.Stream()
    for k in range(3):
        out, st = a.iteration(grid)
        if k in (0, 2):
            got = torch.empty_like(grid)
            graph, kernels = capture(rt, stream, lambda: b.iteration(
                grid, got, stats=False, stream=stream))
            assert rt.cudaGraphDestroy(graph) == 0
            assert st["kernels"] == kernels, (k, st["kernels"], kernels)
            if k == 2:
                break
            # (the captured call has not run: another context for the next ones)
            (_, b), _, _ = contexts(*size, **kw)
            b.iteration(grid, stats=False)
        else:
            b.iteration(grid, stats=False)
        torch.cuda.synchronize()
        grid = out


@pytest.mark.parametrize("kw", [dict(store_scores=True), dict(precision="fp16_split"),
                                dict(model="poisson_fluence", store_scores=True)])
def test_row_pairs_run(kw):
    """The M-step's lists of pairs take three launches (four where some scores are formed again),
    from 2^24 elements of P on: 3328 x 5120 and, just below, 3328 x 4864. Recording goes by the planes."""
    n = []
    for n_data, collect in ((5003, False), (4860, False), (5003, True)):
        (a, _), grid, _ = contexts(16, 60, 4, n_data, 0.15, **kw)
        if collect:
            a.collect(32)
        for _ in range(3):
            out, st = a.iteration(grid)
            grid = out
        assert st["pass1_pruned"] == 1
        n.append(st["kernels"])
    assert n[0] - n[1] in ((3,) if "store_scores" in kw else (3, 4))
    assert n[2] - n[1] == 1  # (the recording itself)


@pytest.mark.parametrize("kw", [dict(), dict(sparse_k=True), dict(precision="fp32"),
                                dict(precision="bf16", sparse_k=True),
                                dict(model="poisson_fluence", sparse_k=True)])
@pytest.mark.parametrize("n_cand", [3, 200])
def test_sparse_iterations(rt, kw, n_cand):  # noqa: F811
    import torch
    (a, b), grid, ds = contexts(16, 30, 2, 300, 0.5, n_cand=n_cand, **kw)
    rng = np.random.default_rng(1)
    cand = np.argsort(rng.random((300, 420)), axis=1)[:, :n_cand].astype(np.int32)
    for ctx in (a, b):
        ctx.set_candidates(torch.as_tensor(cand, device="cuda"))
    _, st = a.sparse_iteration(grid)
    stream = torch.cuda.Stream()
    got = torch.empty_like(grid)
    graph, kernels = capture(rt, stream, lambda: b.sparse_iteration(
        grid, got, stats=False, stream=stream))
    assert rt.cudaGraphDestroy(graph) == 0
    assert st["kernels"] == kernels
