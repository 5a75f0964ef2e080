"""Max pooling past 2^31 rows: more than the flat path's 32-bit rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402


def test_maxpool_special_values_past_2_31_rows():
    """16-byte rows keep their order of maxima where the rows are too many for
    the flat path's 32 bits."""
    planes = 1 << 30
    x = torch.zeros((planes, 2, 4), device=DEV)
    y = torch.empty((planes, 1, 2), device=DEV)
    for p in (0, planes - 1):
        x[p, 0, 1] = float("nan")
        x[p, 0, 2] = 5.0
    k = H.hf_register_kernel(H.MAXPOOL3S2)
    H.hf_launch_single(k, H.maxpool3s2_args(x.view(planes, 1, 2, 4), y.view(planes, 1, 1, 2)), 256)
    torch.cuda.synchronize()
    small = torch.empty((1, 1, 1, 2), device=DEV)
    H.hf_launch_single(k, H.maxpool3s2_args(x[:1].view(1, 1, 2, 4), small), 256)
    torch.cuda.synchronize()
    H.hf_destroy_kernel(k)
    assert H.hf_check_device_error() == 0
    got = torch.stack([y[0, 0], y[planes - 1, 0], small.view(2)]).cpu()
    del x, y
    torch.cuda.empty_cache()
    assert torch.equal(got[0], got[2]) and torch.equal(got[1], got[2])
    assert got[2, 1].item() == 0.0
