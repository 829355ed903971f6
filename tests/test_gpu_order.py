"""GPU: step calls of one context on two streams at a time. Expansions share scratch of the
context, and so do updates: each kind runs in the order of the calls. An expansion and an
update share nothing, and overlap.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def context(precision, model="poisson", **kw):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 32)
    quat, w = emc.quat_generate(4)
    ctx = emc.Context(32, det.q, quat, w, 5300, precision=precision, model=model, w_floor=1e-6, **kw)
    K = np.random.default_rng(2).poisson(0.5, size=(5300, det.q.shape[0])).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    return ctx, quat.shape[0]


def models(n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(5)
    return [torch.rand(32, 32, 32, generator=g, device="cuda") + 0.1 for _ in range(n)]


@pytest.mark.parametrize("model,precision", [("poisson", "bf16_split"), ("poisson", "fp32"),
                                             ("poisson_fluence", "bf16_split"),
                                             ("gaussian", "fp16_split")])
def test_expansions_on_two_streams(model, precision):
    import torch
    ctx, n = context(precision, model)
    grids = models(2)
    want = [ctx.expand(g, 0, n) for g in grids]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for i in range(6):
        with torch.cuda.stream(streams[i % 2]):
            got.append(ctx.expand(grids[i % 2], 0, n, stream=streams[i % 2]))
    torch.cuda.synchronize()
    for i, (L, bias) in enumerate(got):
        assert torch.equal(L, want[i % 2][0]) and torch.equal(bias, want[i % 2][1])
    assert ctx.status() == 0


@pytest.mark.parametrize("precision", ["bf16_split", "fp32"])
def test_expansion_and_update_overlap(precision):
    """An expansion made after an update that still waits on its own stream finishes first;
    both give what they give alone."""
    import torch
    ctx, n = context(precision)
    grid = models(1)[0]
    b = ctx.buffer_sizes(n)
    P = torch.zeros((b.rows, ctx.ld_data), device="cuda")
    P[torch.arange(n, device="cuda"), torch.arange(n, device="cuda") % 5300] = 0.75
    if precision != "fp32":
        P = torch.stack([P.to(torch.bfloat16), torch.zeros_like(P).to(torch.bfloat16)])
    P = P.contiguous().view(torch.uint8).reshape(-1)
    L0, bias0 = ctx.expand(grid, 0, n)
    Num0, den0 = ctx.update(P, n)
    L, bias = ctx.expand(grid, 0, n)
    Num, den = ctx.update(P, n)
    for x in (L, bias, Num, den):
        x.zero_()
    torch.cuda.synchronize()
    from paper_1409_4256_gb300 import emc
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    updated, expanded = torch.cuda.Event(), torch.cuda.Event()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(1_500_000_000)  # cycles: most of a second
    emc._check(emc.lib().emc_update(ctx.h, P.data_ptr(), n, Num.data_ptr(), den.data_ptr(),
                                    s1.cuda_stream), "emc_update")
    updated.record(s1)
    emc._check(emc.lib().emc_expand(ctx.h, grid.data_ptr(), 0, n, L.data_ptr(), bias.data_ptr(),
                                    s2.cuda_stream), "emc_expand")
    expanded.record(s2)
    expanded.synchronize()
    assert not updated.query()
    torch.cuda.synchronize()
    assert torch.equal(L, L0) and torch.equal(bias, bias0)
    assert torch.equal(Num[:n], Num0[:n]) and torch.equal(den[:n], den0[:n])
    assert ctx.status() == 0
