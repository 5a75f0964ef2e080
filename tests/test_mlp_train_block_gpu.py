"""The training kernel of one block, which runs where the cluster of eight does
not fit: the cluster's results bit for bit, from any number of earlier steps."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import costmodel as CM  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402


@pytest.mark.parametrize("batch", [1, 3, 32, 33, 64])
def test_same_bits_as_the_cluster(batch):
    g = torch.Generator().manual_seed(batch)
    X, Y = torch.rand(200, 24, generator=g).to(DEV), torch.rand(200, generator=g).to(DEV)
    idx = torch.randint(0, 200, (5 * batch,), generator=g, dtype=torch.int32).to(DEV)
    out = []
    for train in (H.hf_mlp_train, H.hf_mlp_train_block):
        P = CM.xavier_params(batch).to(DEV)
        M, V = torch.full_like(P, 1e-3), torch.full_like(P, 1e-5)
        loss, grad = torch.empty(5, device=DEV), torch.empty_like(P)
        train(P, M, V, X, Y, idx, 5, batch, t0=7, loss_out=loss, grad_out=grad)
        torch.cuda.synchronize()
        out.append((P, M, V, loss, grad))
    for a, b in zip(*out):
        assert torch.equal(a, b)
    for bad in (dict(steps=-1), dict(batch=65), dict(batch=0)):
        with pytest.raises(H.HFError):
            H.hf_mlp_train_block(P, M, V, X, Y, idx, **{"steps": 1, "batch": batch, **bad})
