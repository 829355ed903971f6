"""GPU: the MLP's forward pass at batches beyond what a grid holds in its second
dimension (65535 blocks of 8 and of 32 rows): the last and a middle stretch of rows get
the bits of a small batch of their own (no row's sums depend on the batch).
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [524416, 2097280, 2097153])  # the last not by tensor cores
def test_large_batches(B):
    import torch
    from paper_1409_4256_gb300 import emc
    n_out, ld = 10, 64
    g = torch.Generator(device="cuda").manual_seed(3)
    params = 0.06 * torch.randn(emc.mlp_param_count(n_out), generator=g, device="cuda")
    X = torch.rand(B, 512, generator=g, device="cuda")

    def forward(x):
        work = torch.empty(emc.mlp_work_size(n_out, x.shape[0]), dtype=torch.uint8, device="cuda")
        z = torch.zeros(x.shape[0], ld, device="cuda")
        emc.mlp_forward(n_out, params, x, x.shape[0], work, z)
        torch.cuda.synchronize()
        return z[:, :n_out]

    z = forward(X)
    few = 128 if B % 128 == 0 else 97  # of the same path
    for at in (B - few, 524288 - 64, B // 2):
        assert torch.equal(forward(X[at:at + few].contiguous()), z[at:at + few])
