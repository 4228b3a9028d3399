"""The largest batches an int holds: their number of tiles must not overflow.
Constant samples, so the mean gradient and loss are those of one sample; they
are summed in binary32, 7 million additions to a chain, so only a bound of
half the value is asked (an overflow gives zeros)."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.slow
def test_largest_batch(sr):
    B, dims = 2 ** 31 - 1, (1, 1, 2)  # 26 GB of samples and targets
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 26 GB of device memory")
    p = np.array([0.5, 0.1, 0.7, 0.2, 0.4, -0.3, 0.1, -0.1], np.float32)
    assert p.size == omlp.param_count(dims)
    x, q = np.array([[1.0]], np.float32), np.array([[0.25, 0.75]], np.float32)
    X = torch.full((B, 1), 1.0, dtype=torch.float32, device="cuda")
    Q = torch.empty((B, 2), dtype=torch.float32, device="cuda")
    Q[:, 0], Q[:, 1] = 0.25, 0.75
    m = sr.MLP(*dims)
    m.set_params(p)
    loss = torch.zeros((), dtype=torch.float32, device="cuda")
    grad = torch.zeros(m.P, dtype=torch.float32, device="cuda")
    m.train_step(X, Q, 0.0, loss=loss, grad=grad)
    torch.cuda.synchronize()
    want = omlp.grad(p, x, q, dims)
    assert np.max(np.abs(grad.cpu().numpy() - want)) <= 0.5 * np.max(np.abs(want))
    assert abs(float(loss.item()) - omlp.loss(p, x, q, dims)) <= 0.5 * omlp.loss(p, x, q, dims)
    m.close()
    del X, Q
    torch.cuda.empty_cache()
