"""GPU: the M-step from the rows' lists of non-zero pairs. A row's list holds 64, a
128-row tile's lists 1024; tiles with more take the planes of P through the tensor cores.
Eq. 2.11 by emc_update against FP64 sums, and iterations against the same
iterations while responsibilities are recorded, which go through the planes.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16_split", "fp16_split"])
@pytest.mark.parametrize("n_data", [5003, 200])  # by pairs; below the rule's line, by planes
def test_update_around_the_limits(precision, n_data):
    """Of three tiles one has rows of at most 8 entries and one row of 64, one a row of 65,
    one rows of up to 60 and far more than 1024 in all. The sums have at most 2 n + 1 exact products (n pairs; hi and lo planes) of one sign,
    each addition off by at most 2^-23 of its result: 2 (n + 1) 2^-23 of the sum."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 16)
    quat, w = emc.quat_generate(4)
    n_rot, n_pix = quat.shape[0], det.q.shape[0]
    ctx = emc.Context(16, det.q, quat, w, n_data, precision=precision)
    rng = np.random.default_rng(5)
    K = rng.poisson(0.7, size=(n_data, n_pix)).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    b = ctx.buffer_sizes(n_rot)
    row = np.arange(b.rows)
    tile = row // 128
    n = np.where(tile % 3 == 2, rng.choice([0, 1, 8, 60], size=b.rows),
                 rng.choice([0, 1, 2, 7, 8], size=b.rows))
    n[(tile % 3 == 0) & (row % 128 == 5)] = 64
    n[(tile % 3 == 1) & (row % 128 == 77)] = 65
    n[n_rot:] = 0
    P = np.zeros((b.rows, ctx.ld_data), dtype=np.float32)
    for j in range(n_rot):
        P[j, rng.permutation(n_data)[:n[j]]] = 0.01 + rng.random(n[j])
    scale, dt = (2.0 ** 14, torch.float16) if precision == "fp16_split" else (1.0, torch.bfloat16)
    x = torch.as_tensor(P, device="cuda") * scale
    hi = x.to(dt)
    lo = (x - hi.float()).to(dt)
    planes = torch.stack([hi, lo]).contiguous()
    held = ((hi.double() + lo.double()) / scale).cpu().numpy()
    assert planes.numel() * 2 == b.prob_bytes
    Num, den = ctx.update(planes.view(torch.uint8).reshape(-1), n_rot)
    want = held[:n_rot, :n_data] @ K.astype(np.float64)
    tol = 2.0 * (n[:n_rot, None] + 1) * 2.0 ** -23
    num = Num[:n_rot, :n_pix].double().cpu().numpy()
    assert np.all(np.abs(num - want) <= tol * want)
    wden = held[:n_rot].sum(1)
    assert np.all(np.abs(den[:n_rot].double().cpu().numpy() - wden) <= tol[:, 0] * wden)
    assert ctx.status() == 0


@pytest.mark.parametrize("model,precision,stored,D,photons,chunk", [
    ("poisson", "bf16_split", True, 60, 400, 0),
    ("poisson", "fp16_split", True, 60, 400, 0),
    ("poisson", "bf16_split", False, 70, 400, 0),    # every live tile's scores kept
    ("poisson", "fp16_split", False, 60, 30, 0),     # some live tiles contracted again
    ("poisson", "bf16_split", True, 60, 400, 2560),  # one chunk above the rule's line, one below
    ("poisson_fluence", "bf16_split", True, 60, 400, 0),
    ("poisson_fluence", "bf16_split", False, 60, 400, 0),
    ("gaussian", "fp16_split", True, 60, 400, 0)])
def test_iteration_equals_planes(model, precision, stored, D, photons, chunk):
    """Three of four frames show a rotation of the first 128, so that tile is over; the
    others leave tiles with short rows. FP32 order of the M-step: 1e-6 relative L2."""
    import torch
    from oracle import oracle
    from paper_1409_4256_gb300 import emc, synth
    n_data = 11003 if chunk else 5303
    quat, w = emc.quat_generate(4)
    rng = np.random.default_rng(9)
    at = np.where(rng.random(n_data) < 0.75, rng.integers(0, 128, n_data),
                  rng.integers(0, quat.shape[0], n_data))
    ds = synth.make_dataset(16, D, n_data, photons / (0.7 * D * D), radius=4.0,
                            rot_true=oracle.quat_to_matrix(quat[at]),
                            fluence_sigma=0.0 if model == "poisson" else 0.2)
    kw = dict(precision=precision, model=model, store_scores=stored, rot_chunk=chunk)
    if model == "gaussian":
        kw["sigma"] = 3.0
    else:
        kw["w_floor"] = 1e-10 * float(ds.model_start.mean())
    a = emc.Context(16, ds.q, quat, w, n_data, **kw)
    if model == "gaussian":  # (not recorded; small chunks of rotations go through the planes)
        kw["rot_chunk"] = 1280
    d = emc.Context(16, ds.q, quat, w, n_data, **kw)
    if model != "gaussian":
        d.collect(32)
    K = torch.as_tensor(ds.K, device="cuda")
    a.set_frames(K)
    d.set_frames(K)
    g = torch.as_tensor(ds.model_start.astype(np.float32), device="cuda")
    for _ in range(3):
        out, st = a.iteration(g)
        ref, _ = d.iteration(g)
        assert st["device_status"] == 0
        rel = float((out.double() - ref.double()).norm() / ref.double().norm())
        assert rel <= 1e-6
        g = ref
    if photons < 400:  # more live tiles than the last L's buffer has places for
        assert st["pass1_exact"] > 2 * 2 * a.sizes_all.rows * a.ld_pix // (4 * 33792)
    if model == "gaussian" or photons < 400:
        return
    tidx, tprob = d.collected_targets(32)
    rows = torch.bincount(tidx[tprob > 0].long(), minlength=a.sizes_all.rows).view(-1, 128)
    over = (rows.amax(1) > 64) | (rows.sum(1) > 1024)
    assert bool(over.any()) and bool((~over & (rows.sum(1) > 0)).any())


@pytest.mark.parametrize("precision", ["bf16_split", "fp32"])
def test_updates_on_several_streams(precision):
    """emc_update takes scratch of the context: calls on two streams at a time give what
    the same calls give one after the other, bit for bit."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 16)
    quat, w = emc.quat_generate(4)
    n_rot, n_data = quat.shape[0], 5003
    ctx = emc.Context(16, det.q, quat, w, n_data, precision=precision)
    rng = np.random.default_rng(6)
    K = rng.poisson(0.7, size=(n_data, det.q.shape[0])).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    b = ctx.buffer_sizes(n_rot)
    planes = []
    for _ in range(2):
        P = torch.zeros((b.rows, ctx.ld_data), device="cuda")
        for _ in range(2):
            k = torch.as_tensor(rng.integers(0, n_data, n_rot), device="cuda")
            P[torch.arange(n_rot, device="cuda"), k] = torch.as_tensor(
                0.1 + rng.random(n_rot).astype(np.float32), device="cuda")
        if precision != "fp32":
            P = torch.stack([P.to(torch.bfloat16), torch.zeros_like(P).to(torch.bfloat16)])
        planes.append(P.contiguous().view(torch.uint8).reshape(-1))
    want = [ctx.update(P, n_rot) for P in planes]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for i in range(6):
        with torch.cuda.stream(streams[i % 2]):
            got.append(ctx.update(planes[i % 2], n_rot, stream=streams[i % 2]))
    torch.cuda.synchronize()
    for i, (Num, den) in enumerate(got):
        assert torch.equal(Num[:n_rot], want[i % 2][0][:n_rot])
        assert torch.equal(den[:n_rot], want[i % 2][1][:n_rot])
    assert ctx.status() == 0
