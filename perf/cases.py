"""Performance cases of the EMC library: the calls a reconstruction makes, over their sizes.

A reconstruction is a chain of emc_iteration calls on models that change a little from one
to the next; the "iteration" cases run such a chain (on models made beforehand, so that
every pass has the same inputs whatever the last one's rounding). A program that holds its
own buffers makes the step calls ("estep", "mstep"); the learned schedule adds sparse
iterations, network training steps and the ranking of the network's logits. Inputs are
synthetic diffraction frames like those of the package's generator (a particle of Gaussian
atoms, Haar-uniform orientations, Poisson counts, a start model 20% off), made on the GPU
from the seed.
"""
import functools
import math

import torch

from paper_1409_4256_gb300 import emc, synth

DEV = "cuda"
STEPS = 8  # models in a state; passes go through them and back, each near the one before


def _iteration(name, N, n_quat, frames, photons, mask=0.0, model="poisson", precision="bf16_split",
               stored=True, reload=False, dense=False, fluence=0.0):
    return dict(name=name, kind="iteration", N=N, n_quat=n_quat, frames=frames, photons=photons,
                mask=mask, model=model, precision=precision, stored=stored, reload=reload,
                dense=dense, fluence=fluence)


def listed():
    return [
        # the smallest workload: 3240 rotations x 1000 frames, where launches and latency count
        _iteration("iter_32", 32, 4, 1000, 0.5),
        # the benchmark workload: 50100 rotations x 20000 frames of 2812 pixels, scores stored
        _iteration("iter_64", 64, 10, 20000, 1.0, mask=0.1),
        # the 128^3 workload: 204960 rotations x 100000 frames, too many scores to store
        _iteration("iter_128", 128, 16, 100000, 0.3, stored=False),
        # frames of unequal intensity (the 160^3 workload's model) at an in-between size
        _iteration("iter_fluence_96", 96, 8, 10007, 0.2, model="poisson_fluence", stored=False,
                   fluence=0.3),
        # the paper's own Gaussian noise model with fluence
        _iteration("iter_gauss_64", 64, 6, 4000, 1.0, mask=0.1, model="gaussian",
                   precision="fp16_split", fluence=0.3),
        # the FP32 form that the split forms are judged against
        _iteration("iter_fp32_64", 64, 4, 2000, 1.0, mask=0.1, precision="fp32"),
        # frames loaded from counts and every tile contracted: the first pass over new data,
        # which each refinement level and each new data set pays for
        _iteration("reload_64", 64, 6, 5000, 1.0, mask=0.1, reload=True, dense=True),
        # scoring a model: expansion and log-likelihood of every frame, in rotation blocks
        dict(name="estep_64", kind="estep", N=64, n_quat=8, frames=4999, photons=1.0, mask=0.1,
             precision="bf16_split", block=6400),
        # the other half by step calls: responsibilities, slice update, compression, division
        dict(name="mstep_64", kind="mstep", N=64, n_quat=6, frames=4999, photons=1.0, mask=0.1,
             precision="bf16_split"),
        # a sparse iteration of the learned schedule: 512 candidate rotations a frame
        dict(name="sparse_64", kind="sparse", N=64, n_quat=10, frames=20000, photons=1.0, mask=0.1,
             cand=512, lists=True),
        # a training step of the proposal network on a batch of 512 frames
        dict(name="mlp_train", kind="train", n_out=50100, batch=512, R=32),
        # the network's logits of 2048 frames ranked into candidate sets
        dict(name="rank", kind="rank", n_out=50100, batch=2048, M=512, R=32),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iteration"] * 5 + ["estep", "mstep", "sparse", "train", "rank"])
    if kind == "train":
        return dict(kind=kind, n_out=_logint(rng, 1380, 204960), batch=128 * rng.randint(1, 4),
                    R=rng.choice([16, 32]))
    if kind == "rank":
        n_out = _logint(rng, 1380, 204960)
        return dict(kind=kind, n_out=n_out, batch=_logint(rng, 100, 2048),
                    M=rng.choice([64, 200, 512]), R=rng.choice([8, 32]))
    N = 2 * _logint(rng, 16, 64)
    n_quat = rng.randint(3, 12)
    frames = _logint(rng, 200, 40000)
    most = {"iteration": 1.2e13, "estep": 1.5e12, "mstep": 1.5e12, "sparse": 3e12}[kind]
    while emc.quat_count(n_quat) * frames * (0.78 * N * N) > most:
        if n_quat > 5:
            n_quat -= 1
        else:
            frames = int(0.8 * frames)
    c = dict(kind=kind, N=N, n_quat=n_quat, frames=frames, photons=rng.choice([0.3, 0.5, 1.0]),
             mask=rng.choice([0.0, 0.1]))
    if kind == "sparse":
        return dict(c, cand=rng.choice([128, 256, 512]), lists=rng.random() < 0.7)
    if kind == "mstep":
        return dict(c, precision=rng.choice(["bf16_split", "bf16_split", "fp16_split"]))
    if kind == "estep":
        return dict(c, precision=rng.choice(["bf16_split", "bf16_split", "fp16_split"]),
                    block=rng.choice([1000, 6400, 12800]))
    form = rng.choice(["poisson"] * 4 + ["poisson_fluence", "gaussian", "fp32"])
    if form == "fp32":
        c["n_quat"], c["frames"] = min(n_quat, 5), min(frames, 3000)
        return _drawn(c, precision="fp32")
    if form == "gaussian":
        c["n_quat"], c["frames"] = min(n_quat, 8), min(frames, 8000)
        return _drawn(c, model=form, precision="fp16_split", fluence=0.3)
    if form == "poisson_fluence":
        return _drawn(c, model=form, stored=rng.random() < 0.5, fluence=0.3)
    again = rng.random() < 0.25
    return _drawn(c, stored=rng.random() < 0.7, reload=again, dense=again,
                      precision=rng.choice(["bf16_split", "bf16_split", "fp16_split"]))


def _drawn(c, **kw):
    d = _iteration(None, *(c[k] for k in ("N", "n_quat", "frames", "photons", "mask")), **kw)
    del d["name"]
    return d


# --- inputs ---------------------------------------------------------------------------


@functools.lru_cache(maxsize=4)
def _rotations(n_quat):
    return emc.quat_generate(n_quat)  # the sampling of Eq. 2.7: data, the same for every seed


@functools.lru_cache(maxsize=4)
def _pixels(N, mask):
    return synth.make_detector(N, N, mask).q  # the detector's pixel positions


def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(1000003 * salt + seed)


def _matrices(q):
    """Rotation matrices [n, 3, 3] of unit quaternions [n, 4] (w, x, y, z)."""
    w, x, y, z = q.unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                       -1).reshape(-1, 3, 3)


def _intensity(p, atoms, N):
    ph = (2 * math.pi / N) * (p @ atoms.T)
    return (torch.exp((-4 * math.pi ** 2 / N ** 2) * (p * p).sum(-1))
            * (torch.cos(ph).sum(-1) ** 2 + torch.sin(ph).sum(-1) ** 2))


def _data(c, seed):
    """Frames int32 [frames, pixels], the models [N, N, N] of successive iterations (the start
    model first, 20% off the truth, then nearer), true orientations [frames, 4]."""
    N, n = c["N"], c["frames"]
    g = _gen(seed, 1)
    q = torch.as_tensor(_pixels(N, c["mask"]), dtype=torch.float32, device=DEV)
    d = torch.randn(50, 3, generator=g, device=DEV)
    radius = 8.0 if N <= 32 else N / 4
    atoms = radius * d / d.norm(dim=1, keepdim=True) * torch.rand(50, 1, generator=g,
                                                                 device=DEV) ** (1 / 3)
    true = torch.randn(n, 4, generator=g, device=DEV)
    true = true / true.norm(dim=1, keepdim=True)
    R = _matrices(true)
    phi = torch.ones(n, 1, device=DEV)
    if c.get("fluence"):
        s = c["fluence"]
        phi = torch.exp(s * torch.randn(n, 1, generator=g, device=DEV) - 0.5 * s * s)
    step = max(1, (1 << 24) // q.shape[0])
    K = torch.empty(n, q.shape[0], dtype=torch.int32, device=DEV)
    scale = None
    for a in range(0, n, step):
        lam = _intensity(torch.einsum("kab,ib->kia", R[a:a + step], q), atoms, N)
        if scale is None:
            scale = c["photons"] / lam.mean()
        # the detector saturates at 250 counts
        K[a:a + step] = torch.poisson(lam.mul_(scale * phi[a:a + step]),
                                      generator=g).clamp_(max=250).to(torch.int32)
    ax = torch.arange(N, dtype=torch.float32, device=DEV) - N // 2
    p = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1)
    truth = torch.cat([_intensity(x, atoms, N) for x in p.split(16)]) * scale
    off = 2 * torch.rand(truth.shape, generator=g, device=DEV) - 1
    return K, [truth * (1 + 0.2 * 0.85 ** t * off) for t in range(STEPS)], true


def _floor(model):
    return 1e-10 * float(model.double().mean())


def _candidates(c, true, seed):
    """int32 [frames, M]: the 32 sampled rotations nearest to the frame's orientation, then
    rotations from all over (a dense E-step's best and a network's others)."""
    quat = torch.as_tensor(_rotations(c["n_quat"])[0], dtype=torch.float32, device=DEV)
    n, M, g = quat.shape[0], min(c["cand"], quat.shape[0]), _gen(seed, 2)
    R = min(32, M)
    offs = torch.randperm(n, generator=g, device=DEV)[:M]
    out = []
    for t in true.split(2048):
        near = torch.topk((t @ quat.T).abs(), R).indices
        rest = (torch.randint(n, (t.shape[0], 1), generator=g, device=DEV) + offs) % n
        taken = (rest[:, :, None] == near[:, None, :]).any(-1)
        order = torch.sort(taken.to(torch.int8), dim=1, stable=True).indices
        out.append(torch.cat([near, rest.gather(1, order)[:, :M - R]], 1))
    return torch.cat(out).to(torch.int32).contiguous()


def _context(c, grid, **kw):
    quat, w = _rotations(c["n_quat"])
    return emc.Context(c["N"], _pixels(c["N"], c["mask"]), quat, w, c["frames"],
                       w_floor=_floor(grid), **kw)


def _chunk(c):
    """Rotations per chunk that keep pass 2's buffer below 8 GB (0: all of them)."""
    ld = -(-c["frames"] // 256) * 256
    rows = -(-emc.quat_count(c["n_quat"]) // 128) * 128
    return 0 if 4 * ld * rows <= 8e9 else max(128, int(8e9 // (4 * ld)) // 128 * 128)


def _train_inputs(c, seed):
    g, B, R = _gen(seed, 3), c["batch"], c["R"]
    X = torch.log1p(torch.empty(B, 512, device=DEV).exponential_(1.0, generator=g))
    tidx = torch.stack([torch.randperm(c["n_out"], generator=g, device=DEV)[:R]
                        for _ in range(B)]).to(torch.int32)
    tprob = torch.softmax(3 * torch.randn(B, R, generator=g, device=DEV), 1)
    ld = (c["n_out"] + 63) // 64 * 64
    parts = []
    for fan in (512, 512, 512, c["n_out"]):
        W = torch.zeros(512, (fan + 63) // 64 * 64, device=DEV)
        W[:, :fan] = math.sqrt(2 / 512) * torch.randn(512, fan, generator=g, device=DEV)
        parts += [W.reshape(-1), torch.zeros(W.shape[1], device=DEV)]
    params = torch.cat(parts)
    # moments as training leaves them after a while
    v = 1e-10 * (0.5 + torch.rand(params.shape, generator=g, device=DEV))
    m = 1e-6 * torch.randn(params.shape, generator=g, device=DEV)
    return dict(X=X, tidx=tidx, tprob=tprob, params=params, m=m, v=v, ld=ld)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "train":
        s = _train_inputs(c, seed)
        return dict(s, case=c, grads=torch.zeros_like(s["params"]), step=200,
                    loss=torch.zeros(1, dtype=torch.float64, device=DEV),
                    work=torch.empty(emc.mlp_work_size(c["n_out"], c["batch"]),
                                     dtype=torch.uint8, device=DEV))
    if kind == "rank":
        z, first = _rank_inputs(c, seed)
        cand = torch.empty(c["batch"], c["M"], dtype=torch.int32, device=DEV)
        return dict(case=c, z=z, first=first, cand=cand, out=torch.empty_like(cand))
    K, models, true = _data(c, seed)
    model = models[0]
    s = dict(case=c, grid=model, models=models, passes=0)
    if kind == "iteration":
        s["ctx"] = _context(c, model, precision=c["precision"], model=c["model"],
                            store_scores=c["stored"], dense_estep=c["dense"],
                            rot_chunk=_chunk(c))
        s["out"] = torch.empty_like(model)
        s["ctx"].set_frames(K)
        s["K"] = K if c["reload"] else None
    elif kind == "sparse":
        quat, _ = _rotations(c["n_quat"])
        s["ctx"] = _context(c, model, n_cand=min(c["cand"], quat.shape[0]), sparse_k=c["lists"],
                            rot_chunk=_chunk(c))
        s["out"] = torch.empty_like(model)
        s["ctx"].set_frames(K)
        s["ctx"].set_candidates(_candidates(c, true, seed))
    else:
        ctx = s["ctx"] = _context(c, model, precision=c["precision"])
        ctx.set_frames(K)
        if kind == "mstep":
            n = ctx.cfg.n_rot
            L, bias = ctx.expand(model, 0, n)
            scores = ctx.scores_buffer(n)
            m, t = ctx.loglik(L, bias, n, scores=scores)
            s.update(bias=bias, scores=scores, m=m, s=t)
    return s


def _rank_inputs(c, seed):
    g = _gen(seed, 4)
    ld = (c["n_out"] + 63) // 64 * 64
    z = 2 * torch.randn(c["batch"], ld, generator=g, device=DEV)
    first = torch.stack([torch.randperm(c["n_out"], generator=g, device=DEV)[:c["R"]]
                         for _ in range(c["batch"])]).to(torch.int32)
    return z, first


# --- the calls ------------------------------------------------------------------------


def run(state):
    return _RUN[state["case"]["kind"]](state)


def _next_model(s):
    t = s["passes"] % (2 * STEPS - 2)
    s["passes"] += 1
    return s["models"][min(t, 2 * STEPS - 2 - t)]


def _run_iteration(s):
    if s["K"] is not None:
        s["ctx"].set_frames(s["K"])
    s["ctx"].iteration(_next_model(s), s["out"], stats=False)
    return s["out"]


def _run_sparse(s):
    s["ctx"].sparse_iteration(_next_model(s), s["out"], stats=False)
    return s["out"]


def _run_estep(s):
    ctx, block = s["ctx"], s["case"]["block"]
    n, m, t = ctx.cfg.n_rot, None, None
    for r0 in range(0, n, block):
        nb = min(block, n - r0)
        L, bias = ctx.expand(s["grid"], r0, nb)
        m, t = ctx.loglik(L, bias, nb, m, t, accumulate=r0 > 0)
    nd = s["case"]["frames"]
    return m[:nd] + torch.log(t[:nd])


def _run_mstep(s):
    ctx = s["ctx"]
    n = ctx.cfg.n_rot
    P = ctx.normalize(None, s["bias"], n, s["m"], s["s"], scores=s["scores"])
    Num, den = ctx.update(P, n)
    g_num, g_den = ctx.compress(0, n, Num, den)
    out = ctx.finalize(g_num, g_den, s["grid"])
    return [Num[:n, :ctx.cfg.n_pix], den[:n], out]


def _run_train(s):
    c = s["case"]
    s["loss"].zero_()
    emc.mlp_train_step(c["n_out"], s["params"], s["grads"], s["m"], s["v"], s["step"], 1e-3, s["X"],
                       s["tidx"], s["tprob"], c["batch"], c["R"], s["work"], s["loss"])
    s["step"] += 1
    return [s["loss"].float(), s["params"], s["grads"], s["m"], s["v"]]


def _run_rank(s):
    c = s["case"]
    emc.topm(s["z"], c["batch"], c["n_out"], s["z"].shape[1], c["M"], s["cand"])
    return [s["cand"], emc.merge_candidates(s["first"], s["cand"], c["M"], out=s["out"])]


_RUN = {"iteration": _run_iteration, "sparse": _run_sparse, "estep": _run_estep,
        "mstep": _run_mstep, "train": _run_train, "rank": _run_rank}


def work(case):
    """What a pass cannot do without. Bytes: inputs and outputs once (frames as 16-bit counts,
    which the context holds). Operations: interpolating and, where the pass compresses,
    reducing every slice element (8 corners each), and the contractions over pixels: every
    pair where every pair is contracted, one rotation per frame in the E- and M-step where
    tiles without weight may be left out."""
    c = case
    if c["kind"] == "train":
        n = 3 * (512 * 512 + 512) + 513 * ((c["n_out"] + 63) // 64 * 64)
        mac = c["batch"] * 512 * (3 * 512 + c["n_out"])
        return {"bytes": 4 * (7 * n + c["batch"] * (512 + 2 * c["R"])),
                "flops": 6 * mac - 2 * c["batch"] * 512 * 512 + 12 * n}
    if c["kind"] == "rank":
        return {"bytes": 4 * c["batch"] * (c["n_out"] + 2 * c["M"] + c["R"]),
                "flops": c["batch"] * c["n_out"]}
    pix, rot = _pixels(c["N"], c["mask"]).shape[0], emc.quat_count(c["n_quat"])
    n, grid = c["frames"], c["N"] ** 3
    ep, pp = rot * pix, rot * n * pix
    if c["kind"] == "estep":
        return {"bytes": 2 * n * pix + 4 * grid + 8 * n, "flops": 2 * pp + 24 * ep}
    if c["kind"] == "mstep":
        return {"bytes": 4 * rot * n + 4 * ep + 2 * n * pix + 8 * grid,
                "flops": 2 * n * pix + 20 * ep}
    if c["kind"] == "sparse":
        m = min(c["cand"], rot)
        return {"bytes": 2 * n * pix + 8 * grid + 4 * n * m,
                "flops": 4 * n * m * pix * min(1.0, c["photons"]) + 44 * ep}
    every = c["dense"] or c["model"] == "gaussian" or c["precision"] == "fp32"
    return {"bytes": (6 if c["reload"] else 2) * n * pix + 8 * grid,
            "flops": (2 * pp if every else 2 * n * pix) + 2 * n * pix + 44 * ep}


# --- the same in 64 bits ----------------------------------------------------------------


def exact(case, seed):
    c = case
    if c["kind"] == "train":
        return _exact_train(c, seed)
    if c["kind"] == "rank":
        return None  # indices
    pix, quat = _pixels(c["N"], c["mask"]), _rotations(c["n_quat"])
    pairs = quat[0].shape[0] * c["frames"]
    if pairs * pix.shape[0] > 3e12 or pairs > 1.2e9:
        return None
    K, models, true = _data(c, seed)
    cand = _candidates(c, true, seed) if c["kind"] == "sparse" else None
    lse, out, Num, den = _exact_em(c, K.double(), models[0], cand)
    return {"estep": lse, "mstep": [Num, den, out]}.get(c["kind"], out)


def _corners(R, q, N):
    """Voxel index and weight of the 8 trilinear corners of every R q, corner by corner."""
    p = torch.einsum("jab,ib->jia", R, q) + N / 2
    f = torch.floor(p)
    t, f = p - f, f.long()
    for k in range(8):
        b = [(k >> 2) & 1, (k >> 1) & 1, k & 1]
        w = torch.ones_like(t[..., 0])
        for a in range(3):
            w = w * (t[..., a] if b[a] else 1 - t[..., a])
        i = [(f[..., a] + b[a]).clamp(0, N - 1) for a in range(3)]
        yield (i[0] * N + i[1]) * N + i[2], w


def _exact_em(c, K, model, cand):
    """One pass of Algorithm 2.1: (lse, new model, numerators, denominators)."""
    N, n = c["N"], K.shape[0]
    q = torch.as_tensor(_pixels(N, c["mask"]), device=DEV)
    quat, wj = (torch.as_tensor(a, device=DEV) for a in _rotations(c["n_quat"]))
    R, g, noise = _matrices(quat), model.double().reshape(-1), c.get("model", "poisson")
    floor = 0.0 if noise == "gaussian" else _floor(model)
    nr, step = R.shape[0], max(1, (1 << 24) // q.shape[0])
    S = torch.empty(nr, n, dtype=torch.float64, device=DEV)
    B = torch.empty(nr, 1, dtype=torch.float64, device=DEV)
    A, total = (K * K).sum(1), K.sum(1)
    for a in range(0, nr, step):
        r = slice(a, a + step)
        W = sum(g[i] * w for i, w in _corners(R[r], q, N)).clamp(min=floor)
        lw = torch.log(wj[r])[:, None]
        if noise == "gaussian":
            G = W @ K.T
            S[r] = (torch.where(A > 0, G * G / A.clamp(min=1), 0.0)
                    - (W * W).sum(1, keepdim=True)) / 2 + lw  # sigma = 1
        else:
            B[r] = W.sum(1, keepdim=True)
            if noise == "poisson":
                S[r] = torch.log(W) @ K.T - B[r] + lw
            else:
                S[r] = torch.log(W / B[r]) @ K.T + lw
    if cand is not None:
        inside = torch.zeros(n, nr, dtype=torch.bool, device=DEV)
        inside.scatter_(1, cand.long(), True)
        S.masked_fill_(~inside.T, -math.inf)
    lse = torch.logsumexp(S, 0)
    if c["kind"] == "estep":
        return lse, None, None, None
    P = S.sub_(lse).exp_()
    P[P < 2.0 ** -150] = 0.0  # responsibilities are defined down to FP32's smallest value
    den = P.sum(1)
    whole = c["kind"] == "mstep"
    kept = []
    num_g, den_g = torch.zeros_like(g), torch.zeros_like(g)
    for a in range(0, nr, step):
        r = slice(a, a + step)
        Q = P[r]
        if noise == "gaussian":  # 1 / phi = G / A
            W = sum(g[i] * w for i, w in _corners(R[r], q, N)).clamp(min=0)
            Q = Q * torch.where(A > 0, (W @ K.T) / A.clamp(min=1), 0.0)
        elif noise == "poisson_fluence":
            Q = Q * torch.where(total > 0, B[r] / total.clamp(min=1), 0.0)
        Num = Q @ K
        if whole:
            kept.append(Num)
        for i, w in _corners(R[r], q, N):
            num_g.index_add_(0, i.reshape(-1), (w * Num).reshape(-1))
            den_g.index_add_(0, i.reshape(-1), (w * den[r, None]).reshape(-1))
    out = torch.where(den_g > 0, num_g / den_g, g).reshape(N, N, N)
    return lse, out, torch.cat(kept) if whole else None, den


def _exact_train(c, seed):
    s = _train_inputs(c, seed)
    B, p, o = c["batch"], s["params"].double(), 0
    Ws, bs = [], []
    for ld in (512, 512, 512, s["ld"]):
        Ws.append(p[o:o + 512 * ld].reshape(512, ld).requires_grad_())
        bs.append(p[o + 512 * ld:o + 513 * ld].clone().requires_grad_())
        o += 513 * ld
    h = s["X"].double()
    for W, b in zip(Ws[:3], bs[:3]):
        h = torch.nn.functional.gelu(h @ W + b)
    z = (h @ Ws[3] + bs[3])[:, :c["n_out"]]
    lp = torch.log_softmax(z, 1).gather(1, s["tidx"].long())
    loss = -(s["tprob"].double() * lp).sum() / B
    grads = torch.autograd.grad(loss, [x for W, b in zip(Ws, bs) for x in (W, b)])
    grad = torch.cat([x.reshape(-1) for x in grads])
    m = 0.9 * s["m"].double() + 0.1 * grad
    v = 0.999 * s["v"].double() + 0.001 * grad * grad
    new = p.detach() - 1e-3 * (m / (1 - 0.9 ** 200)) / (torch.sqrt(v / (1 - 0.999 ** 200)) + 1e-8)
    return [loss.detach(), new, grad, m, v]
