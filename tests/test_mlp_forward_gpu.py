"""The scoring kernel at sample counts around its tiles of 32, its two tiles
per block and its grid, with guard values around the scores."""
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


@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 9729, 19457, 29185])
@pytest.mark.parametrize("off", [0, 1])
def test_forward_counts(n, off):
    """Against the oracle, within 1e-5 of the sum of absolute terms (the
    scale of FP32 rounding in three layers of at most 64 terms)."""
    g = torch.Generator().manual_seed(n)
    P = CM.xavier_params(5)
    P[1536:1600] = 0.05
    X = torch.rand(n, 24, generator=g)
    Xd = torch.empty(24 * n + 1, device=DEV)[off: off + 24 * n].view(n, 24).copy_(X)
    y = torch.full((n + 2,), -7.5, device=DEV)
    H.hf_mlp_forward(P.to(DEV), Xd, y[1: n + 1])
    torch.cuda.synchronize()
    assert y[0].item() == -7.5 and y[n + 1].item() == -7.5
    ref = oracle.mlp_forward(P.double().numpy(), X.numpy())
    scale = oracle.mlp_forward(P.double().abs().numpy(), X.abs().numpy())
    assert np.all(np.abs(y[1: n + 1].cpu().double().numpy() - ref) <= 1e-5 * scale + 1e-12)
