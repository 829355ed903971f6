"""GPU: a training step of the MLP at batches where its kernels take other forms than at 512
rows, against the FP64 oracle with the bars that smaller batches are held to: the loss's
gradient in chunks of 512 rows, with few and with many targets a block of columns, 256-column
tiles of the output layer's input gradient (from 1280 rows), 64-row tiles of the hidden
layers (from 2432 rows, whole tiles or not).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("B,n_out,R", [(1280, 300, 1), (1152, 1500, 64), (2560, 300, 8),
                                       (2500, 100, 4)])
def test_loss_and_gradients(B, n_out, R):
    import torch
    from oracle import learned as ol
    from paper_1409_4256_gb300 import emc, learned
    prop = learned.Proposal(n_out)
    rng = np.random.default_rng(B)
    X = rng.uniform(0, 2, size=(B, 512)).astype(np.float32)
    tidx = np.stack([rng.choice(n_out, R, replace=False) for _ in range(B)]).astype(np.int32)
    tprob = rng.random((B, R)).astype(np.float32)
    tprob /= tprob.sum(axis=1, keepdims=True)
    ps, o = [], 0
    flat = prop.params.cpu().numpy().astype(np.float64)
    sizes = [512, 512, 512, prop.ld_out]
    for out in sizes:
        cols = out if out == 512 and len(ps) < 6 else n_out
        ps.append(flat[o:o + 512 * out].reshape(512, out)[:, :cols])
        o += 512 * out
        ps.append(flat[o:o + out][:cols])
        o += out
    work = torch.empty(emc.mlp_work_size(n_out, B), dtype=torch.uint8, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    emc.mlp_train_step(n_out, prop.params, prop.grads, prop.m, prop.v, 1, 1e-3, dev(X), dev(tidx),
                       dev(tprob), B, R, work, loss)
    torch.cuda.synchronize()
    T = ol.dense_targets(tidx, tprob.astype(np.float64), n_out)
    want, gw = ol.mlp_loss_grads(ps, X.astype(np.float64), T)
    want_b, gb = ol.mlp_loss_grads(ps, X.astype(np.float64), T, operand=ol.bf16_round)
    assert abs(loss.item() - want) < 1e-2 * abs(want)
    assert abs(loss.item() - want_b) < 1e-3 * abs(want_b)
    g, o = prop.grads.cpu().numpy().astype(np.float64), 0
    for layer, out in enumerate(sizes):
        for k, rows in ((2 * layer, 512), (2 * layer + 1, 1)):
            got = g[o:o + rows * out].reshape(rows, out)[:, :gw[k].shape[-1]]
            o += rows * out
            assert rel_l2(got, gw[k].reshape(rows, -1)) < 1e-2, k
            assert rel_l2(got, gb[k].reshape(rows, -1)) < 1e-3, k
