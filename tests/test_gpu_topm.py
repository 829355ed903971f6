"""GPU: emc_topm at the edges of its buffer and chunks, bit for bit: the indices of
the values above the M-th largest in index order, then the first equal ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _expected(z, M):
    t = np.sort(z)[::-1][M - 1]
    above = np.nonzero(z > t)[0]
    return np.concatenate([above, np.nonzero(z == t)[0][:M - len(above)]])


@pytest.mark.parametrize("n,M,pad", [(1, 1, 0), (9, 9, 3), (4095, 1, 1), (4096, 4096, 0),
                                     (4097, 512, 7), (8192, 512, 0), (8193, 4096, 3),
                                     (12289, 3000, 1), (12288, 4097, 0), (30011, 33, 5),
                                     (100003, 512, 1)])
def test_topm_edges(n, M, pad):
    import torch
    from paper_1409_4256_gb300 import emc
    rng = np.random.default_rng(n + M)
    z = np.empty((7, n + pad), dtype=np.float32)
    z[0] = rng.normal(size=n + pad)
    z[1] = np.arange(n + pad)                      # every value enters
    z[2] = -np.arange(n + pad)                     # none after the buffer is full
    z[3] = 0.25                                    # ties only
    z[4] = rng.integers(-3, 4, size=n + pad)       # long ties at the cut
    z[5] = np.where(rng.random(n + pad) < 0.001, rng.random(n + pad), 0)  # mostly exact zeros
    z[6] = np.where(rng.random(n + pad) < 0.5, -np.inf, rng.normal(size=n + pad))
    z[:, n:] = np.inf                              # beyond the first n: not looked at
    cand = torch.full((7, M), -1, dtype=torch.int32, device="cuda")
    emc.topm(torch.as_tensor(z, device="cuda"), 7, n, n + pad, M, cand)
    got = cand.cpu().numpy()
    for b in range(7):
        assert np.array_equal(got[b], _expected(z[b, :n], M)), b
