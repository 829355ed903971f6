"""GPU: emc_topm with few and with many short rows, which take different kernels: the same
indices, bit for bit those of a sort."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,M", [(100, 100), (129, 7), (1380, 64), (4097, 4000), (9000, 4096)])
def test_many_rows_equal_few(n, M):
    import torch
    from paper_1409_4256_gb300 import emc
    rng = np.random.default_rng(n)
    z = rng.standard_normal((1500, n)).astype(np.float32)
    z[::3] = np.round(z[::3]) + 0.0  # ties at the cut (no -0.0, which ranks below 0.0)
    z[5] = 0.0
    order = np.argsort(-z, axis=1, kind="stable")[:, :M]
    t = np.take_along_axis(z, order[:, -1:], 1)
    dev = torch.as_tensor(z, device="cuda")
    for rows in (1500, 40):
        cand = torch.empty(rows, M, dtype=torch.int32, device="cuda")
        emc.topm(dev, rows, n, n, M, cand)
        got = cand.cpu().numpy()
        for b in range(rows):  # above the cut in index order, then the first equal ones
            above = np.nonzero(z[b] > t[b])[0]
            ties = np.nonzero(z[b] == t[b])[0][:M - len(above)]
            assert np.array_equal(got[b], np.concatenate([above, ties])), b
