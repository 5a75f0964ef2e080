"""Batch-norm statistics whose runs are not 16-byte multiples (or whose input
is not aligned): runs shorter than a warp, tiles that end inside a run, one
value, and the bits of every launch shape."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV, check_bn, single  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402
from paper_2007_01277_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (700, 3, 1, 3), (64, 5, 7, 7), (3, 2, 1, 2049), (2, 3, 75, 75),
                                   (41, 2, 5, 10), (1, 300, 1, 5), (9, 1, 17, 31)])
@pytest.mark.parametrize("off", [0, 1])
def test_ragged_runs(shape, off):
    x = W.bn_input(shape, seed=sum(shape))
    xd = torch.empty(x.numel() + 1, device=DEV)[off: off + x.numel()].view(shape).copy_(x)
    ws = H.bn_stats_workspace(xd)
    ref = None
    for threads, grid in ((256, 0), (32, 1), (1024, 2), (96, 50)):
        m, v = torch.empty(shape[1], device=DEV), torch.empty(shape[1], device=DEV)
        single(H.BN_STATS, H.bn_stats_args(xd, m, v, ws), threads, grid)
        torch.cuda.synchronize()
        if ref is None:
            ref = (m, v)
            check_bn(x, m, v)
        assert torch.equal(m, ref[0]) and torch.equal(v, ref[1])
    assert H.hf_check_device_error() == 0
