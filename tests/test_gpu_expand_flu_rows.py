"""GPU: the Poisson-fluence and Gaussian expansions of small blocks of rotations, one launch
with a CTA per rotation (384 threads up to 512 rows, 128 above), give the bits of the whole
sampling, which runs on the tile kernels. Around a slice of 256 columns, the 16 and 40
slices the forms take, and one more; pixels at the grid's edge; a grid beyond the cell layout.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["poisson_fluence", "gaussian"])
@pytest.mark.parametrize("n_pix,N,edge", [(1, 16, False), (255, 16, False), (256, 17, False),
                                          (3001, 32, True), (900, 260, False),
                                          (4095, 64, False), (4096, 64, False),
                                          (10239, 64, False), (10240, 64, False)])
def test_blocks_equal_whole(n_pix, N, edge, model):
    import torch
    from paper_1409_4256_gb300 import emc
    rng = np.random.default_rng(n_pix)
    d = rng.standard_normal((n_pix, 3))
    r = (N / 2 - (0.01 if edge else 1.5)) * rng.random((n_pix, 1)) ** (1 / 3)
    q = r * d / np.linalg.norm(d, axis=1, keepdims=True)
    quat, w = emc.quat_generate(6)
    n = quat.shape[0]
    ctx = emc.Context(N, q, quat, w, 8, model=model, w_floor=1e-6)
    ctx.set_frames(torch.ones(8, n_pix, dtype=torch.int32, device="cuda"))
    g = torch.Generator(device="cuda").manual_seed(N)
    grid = torch.rand(N, N, N, generator=g, device="cuda") + 0.01
    L, bias = ctx.expand(grid, 0, n)
    rows = ctx.sizes_all.rows
    whole, wb = L.view(torch.int16).view(3, rows, ctx.ld_pix), bias.view(-1, rows)
    for r0, nb in ((0, 1), (127, 130), (n - 512, 512), (4001, 513), (300, 1500), (5000, 4096)):
        Lb, bb = ctx.expand(grid, r0, nb)
        rb = (nb + 127) // 128 * 128
        part, bb = Lb.view(torch.int16).view(3, rb, ctx.ld_pix), bb.view(-1, rb)
        assert torch.equal(part[:, :nb], whole[:, r0:r0 + nb])
        assert torch.equal(bb[:, :nb], wb[:, r0:r0 + nb])
        assert int(part[:, nb:].count_nonzero()) == 0
        assert bool(torch.isneginf(bb[0, nb:]).all()) and int(bb[1:, nb:].count_nonzero()) == 0
    assert ctx.status() == 0
