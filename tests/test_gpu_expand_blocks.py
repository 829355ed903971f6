"""GPU: the expansion gives the same bits whatever the block of rotations it runs
over: a whole sampling (32 rotations a CTA), and blocks small enough for 16 a CTA,
starting and ending inside row tiles. Interior pixels (cell layout), an odd grid,
pixels at the grid's edge (bounds-checked corners) and a grid beyond the cell
layout's 256^3.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,edge,precision", [(32, False, "bf16_split"), (33, False, "fp16_split"),
                                              (32, True, "bf16_split"), (32, False, "fp32"),
                                              (260, False, "bf16_split")])
def test_blocks_equal_whole(N, edge, precision):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(32, 32)
    q = det.q * ((N / 2 - 0.01) / 15.0 if edge else 1.0)
    quat, w = emc.quat_generate(6)
    n = quat.shape[0]
    ctx = emc.Context(N, q, quat, w, 8, precision=precision, w_floor=1e-6)
    g = torch.Generator(device="cuda").manual_seed(N)
    grid = torch.rand(N, N, N, generator=g, device="cuda") + 0.01

    def planes(L, rows):
        t = torch.float32 if precision == "fp32" else torch.int16
        return L.view(t).view(-1, rows, ctx.ld_pix)

    L, bias = ctx.expand(grid, 0, n)
    whole = planes(L, ctx.sizes_all.rows)
    for r0, nb in ((0, 1), (127, 130), (4001, 700), (n - 33, 33)):
        Lb, bb = ctx.expand(grid, r0, nb)
        rows = (nb + 127) // 128 * 128
        part = planes(Lb, rows)
        assert torch.equal(part[:, :nb], whole[:, r0:r0 + nb])
        assert torch.equal(bb[:nb], bias[r0:r0 + nb])
        assert int(part[:, nb:].count_nonzero()) == 0 and bool(torch.isinf(bb[nb:]).all())
    assert ctx.status() == 0


@pytest.mark.parametrize("model,precision", [("poisson_fluence", "bf16_split"),
                                             ("gaussian", "fp16_split")])
def test_blocks_equal_whole_other_models(model, precision):
    """The Poisson-fluence expansion keeps W in a buffer of rot_chunk rotations, so a
    whole sampling runs in several pieces there; the Gaussian one has its own layout."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(32, 32)
    quat, w = emc.quat_generate(6)
    n = quat.shape[0]
    K = torch.ones(8, det.q.shape[0], dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(7)
    grid = torch.rand(32, 32, 32, generator=g, device="cuda") + 0.01
    got = []
    for chunk, block in ((0, n), (1000, n), (256, 777)):
        ctx = emc.Context(32, det.q, quat, w, 8, precision=precision, model=model, w_floor=1e-6,
                          rot_chunk=chunk)
        ctx.set_frames(K)
        planes, bias = [], []
        for r0 in range(0, n, block):
            nb = min(block, n - r0)
            L, b = ctx.expand(grid, r0, nb)
            rows = (nb + 127) // 128 * 128
            part = L.view(torch.int16).view(3, rows, ctx.ld_pix)
            assert int(part[:, nb:].count_nonzero()) == 0
            planes.append(part[:, :nb])
            bias.append(b.view(-1, rows)[:, :nb])
        assert ctx.status() == 0
        got.append((torch.cat(planes, 1), torch.cat(bias, 1)))
    for planes, bias in got[1:]:
        assert torch.equal(planes, got[0][0]) and torch.equal(bias, got[0][1])
