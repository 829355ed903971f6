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
