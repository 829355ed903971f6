"""GPU: the step calls and the alignment of what the caller hands over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ERR_ARG = -1


def context(N=16, D=14, n_quat=2, n_data=300, **kw):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(D, N)
    quat, w = emc.quat_generate(n_quat)
    ctx = emc.Context(N, det.q, quat, w, n_data, w_floor=1e-6, **kw)
    K = np.random.default_rng(1).poisson(0.7, size=(n_data, det.q.shape[0])).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    return ctx, quat.shape[0]


@pytest.mark.parametrize("precision,D,n_quat,n_data", [
    ("bf16_split", 14, 2, 300), ("bf16_split", 60, 4, 5300),  # by planes, by pairs
    ("fp16_split", 60, 4, 5300), ("bf16", 14, 2, 300), ("fp32", 14, 2, 300)])
def test_update_refuses_what_it_cannot_read(precision, D, n_quat, n_data):
    import torch
    from paper_1409_4256_gb300 import emc
    ctx, n = context(16, D, n_quat, n_data, precision=precision)
    b = ctx.buffer_sizes(n)
    P = torch.zeros(b.prob_bytes + 16, dtype=torch.uint8, device="cuda").data_ptr()
    Num = torch.zeros(b.num_bytes + 16, dtype=torch.uint8, device="cuda").data_ptr()
    den = torch.zeros(b.rows, device="cuda").data_ptr()
    call = emc.lib().emc_update
    assert call(ctx.h, P, n, Num, den, 0) == 0
    for off in (2, 4, 8):
        assert call(ctx.h, P + off, n, Num, den, 0) == ERR_ARG
        assert call(ctx.h, P, n, Num + off, den, 0) == ERR_ARG
    torch.cuda.synchronize()
    assert ctx.status() == 0


@pytest.mark.parametrize("lists", [True, False])
def test_sparse_update_takes_any_float_address(lists):
    """Num at 4, 8 and 12 bytes past a 16-byte boundary: the numbers of an aligned one. One
    frame a pair's row at most twice, so no sum depends on the order of its atomics."""
    import torch
    from paper_1409_4256_gb300 import emc
    ctx, n = context(precision="bf16_split", n_cand=4, sparse_k=lists, n_data=200)
    b = ctx.sizes_all
    cand = torch.arange(800, dtype=torch.int32, device="cuda").remainder(n).view(200, 4)
    ctx.set_candidates(cand.contiguous())
    P = torch.zeros((ctx.ld_data, 4), device="cuda")
    P[:200] = 0.25
    P[:200, 1] = 0.0
    want, wden = ctx.sparse_update(P)
    for off in (1, 2, 3):
        buf = torch.full((b.rows * b.ld_pix + 4,), -1.0, device="cuda")
        den = torch.empty(b.rows, device="cuda")
        emc._check(emc.lib().emc_sparse_update(ctx.h, P.data_ptr(), buf.data_ptr() + 4 * off,
                                               den.data_ptr(), 0), "emc_sparse_update")
        torch.cuda.synchronize()
        assert torch.equal(buf[off:off + want.numel()].view_as(want), want)
        assert bool((buf[:off] == -1).all()) and bool((buf[off + want.numel():] == -1).all())
        assert torch.equal(den, wden)
    assert ctx.status() == 0


@pytest.mark.parametrize("model,precision", [("poisson_fluence", "bf16_split"),
                                             ("gaussian", "fp16_split")])
@pytest.mark.parametrize("D", [14, 40])
def test_expansion_takes_any_plane_address(model, precision, D):
    """L of the models whose planes were written one element at a time, at 2, 4 and 6 bytes
    past an 8-byte boundary: the bits of an aligned one."""
    import torch
    from paper_1409_4256_gb300 import emc
    ctx, n = context(D=D, model=model, precision=precision)
    g = torch.Generator(device="cuda").manual_seed(2)
    grid = torch.rand(16, 16, 16, generator=g, device="cuda") + 0.1
    L, bias = ctx.expand(grid, 0, n)
    for off in (1, 2, 3):
        buf = torch.full((L.numel() // 2 + 4,), -1, dtype=torch.int16, device="cuda")
        got = torch.empty_like(bias)
        emc._check(emc.lib().emc_expand(ctx.h, grid.data_ptr(), 0, n, buf.data_ptr() + 2 * off,
                                        got.data_ptr(), 0), "emc_expand")
        torch.cuda.synchronize()
        assert torch.equal(buf[off:off + L.numel() // 2], L.view(torch.int16))
        assert bool((buf[:off] == -1).all()) and bool((buf[off + L.numel() // 2:] == -1).all())
        assert torch.equal(got, bias)
    assert ctx.status() == 0
