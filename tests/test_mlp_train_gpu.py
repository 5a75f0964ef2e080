"""The training kernel at batches that leave lanes, sample groups or whole
warps of a block without work, and over several steps (its buffers alternate
from step to step)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import costmodel as CM  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402


@pytest.mark.parametrize("batch", [1, 3, 4, 16, 33, 63, 64])
def test_train_batches_and_steps(batch):
    """Each step's gradient against the oracle (the tolerance of the one-step
    test at batch 64), and a run of three steps equal, bit for bit, to three
    runs of one step."""
    g = torch.Generator().manual_seed(batch)
    X, Y = torch.rand(200, 24, generator=g), torch.rand(200, generator=g)
    idx = torch.randint(0, 200, (3 * batch,), generator=g, dtype=torch.int32)
    P0 = CM.xavier_params(batch)
    Xd, Yd, idxd = X.to(DEV), Y.to(DEV), idx.to(DEV)
    P, M, V = P0.to(DEV), torch.zeros(5825, device=DEV), torch.zeros(5825, device=DEV)
    losses = []
    for t in range(3):
        before = P.cpu().double().numpy()
        grad, loss = torch.empty(5825, device=DEV), torch.empty(1, device=DEV)
        H.hf_mlp_train(P, M, V, Xd, Yd, idxd[t * batch:], 1, batch, t0=t, loss_out=loss, grad_out=grad)
        torch.cuda.synchronize()
        rows = idx[t * batch: (t + 1) * batch].long().numpy()
        _, g_ref = oracle.mlp_loss_grad(before, X.numpy()[rows], Y.numpy()[rows])
        gg = grad.cpu().double().numpy()
        assert np.all(np.abs(gg - g_ref) <= 1e-4 * np.abs(g_ref).max() + 1e-7)
        losses.append(loss.item())
    P3, M3, V3 = P0.to(DEV), torch.zeros(5825, device=DEV), torch.zeros(5825, device=DEV)
    loss3 = torch.empty(3, device=DEV)
    H.hf_mlp_train(P3, M3, V3, Xd, Yd, idxd, 3, batch, loss_out=loss3)
    torch.cuda.synchronize()
    assert torch.equal(P, P3) and torch.equal(M, M3) and torch.equal(V, V3)
    assert loss3.tolist() == losses
