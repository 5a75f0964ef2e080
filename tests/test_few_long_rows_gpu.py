"""Tensors of few rows too long for a ring of the resampling bodies: a thread
per output below a number of rows per warp, the flat path's items above."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import DEV, check_upsample, single  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402
from paper_2007_01277_gb300 import workloads as W  # noqa: E402

ARGS = {H.UPSAMPLE2X: H.upsample2x_args, H.MAXPOOL3S2: H.maxpool3s2_args, H.IM2COL3: H.im2col3_args}


def _out(body, s):
    shape = {H.UPSAMPLE2X: (s[0], s[1], 2 * s[2], 2 * s[3]), H.IM2COL3: (s[0], 9 * s[1], s[2] * s[3]),
             H.MAXPOOL3S2: (s[0], s[1], (s[2] - 1) // 2 + 1, (s[3] - 1) // 2 + 1)}[body]
    return torch.full(shape, -7.5, device=DEV)


# long rows, and row counts on both sides of each body's line at these grids
@pytest.mark.parametrize("shape", [(1, 1, 1, 508), (1, 1, 2, 545), (1, 1, 1, 1015), (1, 2, 3, 1057), (1, 1, 2, 2305),
                                   (3, 1, 1, 9731), (1, 1, 1, 77825), (1, 1, 5, 15553),
                                   (2, 61, 5, 509), (1, 153, 2, 1025)])
@pytest.mark.parametrize("off", [0, 1])
def test_long_rows(shape, off):
    x, z = W.upsample_input(shape), W.maxpool_input(shape)
    xd, zd = (torch.empty(t.numel() + 1, device=DEV)[off: off + t.numel()].view(shape).copy_(t) for t in (x, z))
    pool, col = oracle.maxpool3s2p1(z.numpy()), oracle.im2col3(z.numpy())
    for threads, grid in ((32, 1), (96, 3), (256, 152), (256, 0)):
        y, p, c = _out(H.UPSAMPLE2X, shape), _out(H.MAXPOOL3S2, shape), _out(H.IM2COL3, shape)
        single(H.UPSAMPLE2X, H.upsample2x_args(xd, y), threads, grid)
        single(H.MAXPOOL3S2, H.maxpool3s2_args(zd, p), threads, grid)
        single(H.IM2COL3, H.im2col3_args(zd, c), threads, grid)
        torch.cuda.synchronize()
        check_upsample(x, y)
        assert np.array_equal(p.cpu().numpy(), pool)
        assert np.array_equal(c.cpu().numpy().ravel(), col.ravel())
    assert H.hf_check_device_error() == 0


@pytest.mark.parametrize("body", list(ARGS))
def test_one_row_uses_every_warp(body):
    """The same values as one row and as a thousand rows, neither of which a
    ring holds, are the same work: the row may not be left to one warp (where it
    took 100 times as long and more)."""
    k = H.hf_register_kernel(body)
    best = []
    for shape in ((1, 1, 1, 1000001), (1, 1, 1000, 1001)):
        x, y = torch.rand(shape, device=DEV), _out(body, shape)
        args = ARGS[body](x, y)
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            H.hf_launch_single(k, args, 256)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        best.append(min(times[1:]))
    H.hf_destroy_kernel(k)
    assert best[0] < 8 * best[1]
