"""The training step at the sizes where its tiles can go wrong: networks of the
smallest, largest and odd widths, batches around a tile of eight samples and
around the number of tiles that get a CTA of their own; gradient and loss
against the FP64 oracle, within the tolerances of test_gpu_mlp.py."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 2), (9, 64, 40), (32, 64, 64), (5, 33, 41), (17, 7, 3)])
def test_gradient_for_widths_and_batches(sr, dims):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for B in (1, 7, 8, 9, 16, 200, 16 * sms, 16 * sms + 3):
        rng = np.random.default_rng(B)
        p = rng.normal(0, 0.3, omlp.param_count(dims)).astype(np.float32)
        X = rng.normal(0, 1, (B, dims[0])).astype(np.float32)
        Q = rng.dirichlet(np.ones(dims[2]) * 0.3, size=B).astype(np.float32)
        m = sr.MLP(*dims)
        m.set_params(p)
        loss = torch.zeros((), dtype=torch.float32, device="cuda")
        grad = torch.full((m.P,), 7.0, dtype=torch.float32, device="cuda")
        m.train_step(torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda(), 0.0, loss=loss, grad=grad)
        torch.cuda.synchronize()
        g_ref = omlp.grad(p, X, Q, dims)
        assert np.max(np.abs(grad.cpu().numpy().astype(np.float64) - g_ref)) <= 2e-4 * np.max(np.abs(g_ref)) + 1e-7, B
        assert float(loss.item()) == pytest.approx(omlp.loss(p, X, Q, dims), rel=2e-5), B
        assert np.array_equal(m.get_params(), p)
        m.close()
