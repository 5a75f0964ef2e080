"""The training kernel at batches that are not multiples of four when an
activation is infinite: samples past the batch add nothing to a gradient."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import costmodel as CM  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402


@pytest.mark.parametrize("batch", [1, 3, 33, 62, 63, 64])
def test_infinite_activation(batch):
    """Unit 5 of layer 2 has an infinite bias and a positive output weight:
    every output and error is infinite, so its output weight's gradient is a
    sum of infinities and nothing else."""
    g = torch.Generator().manual_seed(batch)
    X, Y = torch.rand(70, 24, generator=g).to(DEV), torch.rand(70, generator=g).to(DEV)
    idx = torch.randint(0, 70, (batch,), generator=g, dtype=torch.int32).to(DEV)
    P = CM.xavier_params(3)
    P[5696 + 5] = float("inf")
    P[5760 + 5] = 0.25
    P = P.to(DEV)
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    grad, loss = torch.empty_like(P), torch.empty(1, device=DEV)
    H.hf_mlp_train(P, M, V, X, Y, idx, 1, batch, loss_out=loss, grad_out=grad)
    torch.cuda.synchronize()
    assert grad[5760 + 5].item() == float("inf") and grad[5824].item() == float("inf")
    assert loss.item() == float("inf")
