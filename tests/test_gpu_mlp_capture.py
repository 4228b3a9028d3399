"""A training step captured after an eager one of a smaller batch: batches up to
the next multiple of 16 need no more workspace, so the capture allocates
nothing; replays give the eager step's gradient."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm,batch", [(1, 16), (8, 9), (17, 32), (100, 112), (2400, 2400)])
def test_capture_after_a_smaller_batch(sr, warm, batch):
    dims = (9, 64, 40)
    rng = np.random.default_rng(batch)
    p = rng.normal(0, 0.3, omlp.param_count(dims)).astype(np.float32)
    X = torch.from_numpy(rng.normal(0, 1, (batch, dims[0])).astype(np.float32)).cuda()
    Q = torch.from_numpy(rng.dirichlet(np.ones(dims[2]), size=batch).astype(np.float32)).cuda()
    m, ref = sr.MLP(*dims), sr.MLP(*dims)
    m.set_params(p)
    ref.set_params(p)
    grad, want = (torch.zeros(m.P, dtype=torch.float32, device="cuda") for _ in range(2))
    ref.train_step(X, Q, 0.0, grad=want)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        m.train_step(X[:warm], Q[:warm], 0.0, grad=grad)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        m.train_step(X, Q, 0.0, grad=grad)
    for _ in range(2):
        grad.fill_(7.0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(grad, want)
    m.close()
    ref.close()
