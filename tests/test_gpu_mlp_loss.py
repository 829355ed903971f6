"""GPU: the loss kernels of the MLP's training step at ragged batches, widths and
target counts (more targets than a warp, repeated targets, rows and columns
beyond the CTAs' blocks), from the logits emc_mlp_forward gives for the same
parameters. dL/dz = (softmax(z) sum_r p_r - onehot(p)) / B in FP64; its column
sums are the output bias's gradient. The kernel's FP32 softmax carries the
rounding of z - lse (|z - lse| < 32: 4e-6) and of expf, 1e-5 of each term in all,
and B additions of FP32 at 2^-24 of the terms' sum.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_out,R", [(1, 1, 1), (3, 65, 2), (33, 127, 33), (128, 129, 40),
                                       (600, 64, 5), (640, 300, 32), (1024, 100, 1)])
def test_output_bias_gradient_and_loss(B, n_out, R):
    import torch
    from paper_1409_4256_gb300 import emc
    g = torch.Generator(device="cuda").manual_seed(B + n_out)
    dev = "cuda"
    n, ld = emc.mlp_param_count(n_out), (n_out + 63) // 64 * 64
    params = 0.06 * torch.randn(n, generator=g, device=dev)
    X = torch.rand(B, 512, generator=g, device=dev)
    tidx = torch.randint(n_out, (B, R), generator=g, device=dev, dtype=torch.int32)
    tprob = torch.rand(B, R, generator=g, device=dev)
    work = torch.empty(emc.mlp_work_size(n_out, B), dtype=torch.uint8, device=dev)
    z = torch.zeros(B, ld, device=dev)
    emc.mlp_forward(n_out, params, X, B, work, z)
    zd, p = z[:, :n_out].double(), tprob.double()
    soft = torch.softmax(zd, 1) * p.sum(1, keepdim=True) / B
    dz = soft.clone().scatter_add_(1, tidx.long(), -p / B)
    loss_want = -(p * torch.log_softmax(zd, 1).gather(1, tidx.long())).sum() / B
    grads, m, v = (torch.zeros(n, device=dev) for _ in range(3))
    loss = torch.zeros(1, dtype=torch.float64, device=dev)
    emc.mlp_train_step(n_out, params, grads, m, v, 1, 1e-3, X, tidx, tprob, B, R, work, loss)
    db = grads[n - ld:n - ld + n_out].double()
    tol = 1e-5 * soft.sum(0) + (B + R) * 2.0 ** -24 * (soft.sum(0) + (dz - soft).abs().sum(0))
    assert bool(((db - dz.sum(0)).abs() <= tol + 1e-12).all())
    assert abs(float(loss[0] - loss_want)) <= 1e-5 * float(p.sum()) / B * 32
    assert bool((grads[n - ld + n_out:] == 0).all())
