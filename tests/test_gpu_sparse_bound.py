"""GPU: the sparse E-step from the frames' non-zero lists against FP64 sums of the planes of
log W: short and long lists, few and many pairs a rotation (the forms that sparse.cu
chooses between), rows that its integers cannot hold, an L that is not 4-byte aligned, and
biases far larger than FP32 resolves (a model scaled far above the counts).
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


@pytest.mark.parametrize("precision", ["bf16_split", "fp16_split", "fp32", "bf16"])
@pytest.mark.parametrize("n_pix,entries,M", [
    (700, 90, 200),    # short lists
    (700, 383, 200), (700, 385, 200), (700, 500, 20),  # around the line; few pairs a rotation
    (7040, 400, 200), (7039, 400, 200)])  # one launch or two of the first stage
def test_scores_equal_exact_sums(precision, n_pix, entries, M):
    """S = sum K (hi + mid + lo) + bias is off by the integers' 2^-25 a count at most (plain
    FP64 otherwise), lse by no more; P by twice that, by FP32's rounding of S - lse and by
    its exponential (|x| <= 111: 111 x 2^-23 + 2^-21)."""
    import torch
    from paper_1409_4256_gb300 import emc
    rng = np.random.default_rng(n_pix + entries + M)
    d = rng.standard_normal((n_pix, 3))
    q = 14.0 * rng.random((n_pix, 1)) ** (1 / 3) * d / np.linalg.norm(d, axis=1, keepdims=True)
    quat, w = emc.quat_generate(2)
    n_rot, n_data = quat.shape[0], 150
    ctx = emc.Context(32, q, quat, w, n_data, precision=precision, n_cand=M, sparse_k=True,
                      w_floor=1e-9)
    K = np.zeros((n_data, n_pix), dtype=np.int32)
    for k in range(n_data):
        K[k, rng.permutation(n_pix)[:entries]] = rng.integers(1, 9, entries)
    K[3] = 0
    K[4, :entries + 1] = 1  # (the mean stays `entries` or just misses it)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    cand = np.argsort(rng.random((n_data, n_rot)), axis=1)[:, :M].astype(np.int32)
    ctx.set_candidates(torch.as_tensor(cand, device="cuda"))
    g = torch.Generator(device="cuda").manual_seed(1)
    grid = torch.exp(0.4 * torch.randn(32, 32, 32, generator=g, device="cuda"))
    L, bias = ctx.expand(grid, 0, n_rot)
    P, lse = ctx.sparse_estep(L, bias)
    assert ctx.status() == 0
    rows = ctx.sizes_all.rows
    t = {"fp32": torch.float32, "fp16_split": torch.float16}.get(precision, torch.bfloat16)
    W = L.view(t).view(-1, rows, ctx.ld_pix).double().sum(0)[:n_rot, :n_pix]
    Kd = torch.as_tensor(K, device="cuda").double()
    S = (W @ Kd.T).T + bias[:n_rot]
    S = torch.gather(S, 1, torch.as_tensor(cand, device="cuda").long())
    want = torch.logsumexp(S, 1)
    off = float(Kd.sum(1).max()) * 2.0 ** -25 + 1e-9
    assert float((lse[:n_data] - want).abs().max()) <= off + 2e-6  # (FP32 exponentials in the sum)
    x = S - want[:, None]
    got, ref = P[:n_data].double(), torch.exp(x)
    tol = ref * (2 * off + 2e-6 + 111 * 2.0 ** -23 + 2.0 ** -21) + 2.0 ** -125
    assert bool(((got - ref).abs() <= tol).all())
    # the same from an L at an odd 16-bit address
    if precision != "fp32":
        buf = torch.empty(L.numel() + 2, dtype=torch.uint8, device="cuda")
        buf[2:] = L
        P2, lse2 = torch.empty_like(P), torch.empty_like(lse)
        torch.cuda.synchronize()
        emc._check(emc.lib().emc_sparse_estep(ctx.h, buf.data_ptr() + 2, bias.data_ptr(),
                                              P2.data_ptr(), lse2.data_ptr(), 0), "sparse_estep")
        torch.cuda.synchronize()
        assert torch.equal(P2[:n_data], P[:n_data]) and torch.equal(lse2[:n_data], lse[:n_data])


@pytest.mark.parametrize("entries", [90, 500])
def test_rows_beyond_the_integers(entries):
    """FP32 rows with values of up to 3000: scored from their parts, as before; a row with
    an infinite log W makes its frames' lse non-finite, which is reported."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(30, 32)
    quat, w = emc.quat_generate(2)
    n_pix, n_rot, n_data, M = det.q.shape[0], quat.shape[0], 150, 200
    rng = np.random.default_rng(entries)
    ctx = emc.Context(32, det.q, quat, w, n_data, precision="fp32", n_cand=M, sparse_k=True)
    K = np.zeros((n_data, n_pix), dtype=np.int32)
    for k in range(n_data):
        K[k, rng.permutation(n_pix)[:entries]] = 1
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    cand = np.argsort(rng.random((n_data, n_rot)), axis=1)[:, :M].astype(np.int32)
    ctx.set_candidates(torch.as_tensor(cand, device="cuda"))
    rows = ctx.sizes_all.rows
    L = np.zeros((rows, ctx.ld_pix), dtype=np.float32)
    L[:n_rot, :n_pix] = rng.standard_normal((n_rot, n_pix))
    L[5, :n_pix] *= 1000.0
    L[9, 3] = -200.0
    bias = np.zeros(rows)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    P, lse = ctx.sparse_estep(dev(L), dev(bias))
    assert ctx.status() == 0
    S = np.take_along_axis(K.astype(np.float64) @ L[:n_rot, :n_pix].T.astype(np.float64), cand, 1)
    m = S.max(1, keepdims=True)
    want = (m + np.log(np.exp(S - m).sum(1, keepdims=True)))[:, 0]
    # (FP32 sums of a beyond row: entries roundings of at most 2^-24 of 1000 x entries)
    assert np.all(np.abs(lse[:n_data].cpu().numpy() - want) <= entries ** 2 * 1000.0 * 2.0 ** -24)
    L[7, 0] = np.inf
    ctx.sparse_estep(dev(L), dev(bias))
    assert ctx.status() == (-6 if K[:, 0].any() else 0)


@pytest.mark.parametrize("lists,entries", [(False, 90), (True, 90), (True, 500)])
def test_candidates_outside_the_sampling(lists, entries):
    """An index outside [0, n_rot) is reported and left out: the other pairs' P and lse are
    those of the frame without it, and so are the M-step and the missed mass."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(30, 32)
    quat, w = emc.quat_generate(2)
    n_pix, n_rot, n_data, M = det.q.shape[0], quat.shape[0], 150, 200
    rng = np.random.default_rng(entries)
    ctx = emc.Context(32, det.q, quat, w, n_data, n_cand=M, sparse_k=lists, store_scores=True,
                      w_floor=1e-6)
    K = np.zeros((n_data, n_pix), dtype=np.int32)
    for k in range(n_data):
        K[k, rng.permutation(n_pix)[:entries]] = 1
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    cand = np.argsort(rng.random((n_data, n_rot)), axis=1)[:, :M].astype(np.int32)
    g = torch.Generator(device="cuda").manual_seed(1)
    grid = torch.exp(0.1 * torch.randn(32, 32, 32, generator=g, device="cuda"))
    L, bias = ctx.expand(grid, 0, n_rot)
    ctx.set_candidates(torch.as_tensor(cand, device="cuda"))
    P, lse = ctx.sparse_estep(L, bias)
    assert ctx.status() == 0
    bad = cand.copy()
    out = rng.random(cand.shape) < 0.1
    bad[out] = rng.choice([-1, -(2 ** 31), n_rot, 2 ** 31 - 1], size=int(out.sum()))
    ctx.set_candidates(torch.as_tensor(bad, device="cuda"))
    assert ctx.status() == -1
    Pb, lseb = ctx.sparse_estep(L, bias)
    Num, den = ctx.sparse_update(Pb)
    assert ctx.status() == 0
    off = torch.as_tensor(out, device="cuda")
    S = torch.log(P[:n_data].double()) + lse[:n_data, None]
    want = torch.logsumexp(torch.where(off, -torch.inf, S), 1)
    assert float((lseb[:n_data] - want).abs().max()) <= 1e-5
    assert bool((Pb[:n_data][off] == 0).all())
    assert float((Pb[:n_data].double().sum(1) - 1).abs().max()) <= 1e-5
    assert abs(float(den[:n_rot].double().sum()) - n_data) <= 1e-5 * n_data
    ctx.iteration(grid)
    missed = ctx.missed_mass()
    fr = torch.arange(n_data, dtype=torch.int32, device="cuda")
    dense = ctx.responsibilities(fr).double()
    held = torch.gather(dense, 1, torch.as_tensor(cand, device="cuda").long())
    left = 1 - torch.where(off, 0.0, held).sum(1)
    assert float((missed.double() - left).abs().max()) <= 1e-6
    assert ctx.status() == 0
