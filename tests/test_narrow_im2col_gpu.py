"""im2col on intervals of one and two warps: its strips there, the kernels
compiled with them and without, and the shapes that stay on the flat path."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402
from paper_2007_01277_gb300 import workloads as W  # noqa: E402


def _other(body):
    """A small kernel of `body` to fuse with."""
    x = torch.rand(2, 3, 20, 24, device=DEV)
    if body == H.BN_STATS:
        m, v, ws = torch.empty(3, device=DEV), torch.empty(3, device=DEV), H.bn_stats_workspace(x)
        return H.bn_stats_args(x, m, v, ws), (x, m, v, ws)
    if body == H.HIST256:
        x = W.hist_input(5000).to(DEV)
        b = torch.zeros(256, dtype=torch.int32, device=DEV)
        return H.hist256_args(x, b), (x, b)
    y = torch.empty((2, 3, 40, 48) if body == H.UPSAMPLE2X else (2, 3, 10, 12), device=DEV)
    return (H.upsample2x_args if body == H.UPSAMPLE2X else H.maxpool3s2_args)(x, y), (x, y)


@pytest.mark.parametrize("shape,off", [((2, 3, 30, 56), 0), ((1, 4, 15, 64), 0), ((3, 2, 29, 60), 0), ((3, 2, 29, 60), 1),
                                       ((2, 2, 14, 52), 0), ((4, 3, 7, 7), 0), ((1, 1, 1, 64), 0)])
def test_narrow_intervals(shape, off):
    x = W.im2col_input(shape)
    xd = torch.empty(x.numel() + 1, device=DEV)[off: off + x.numel()].view(shape).copy_(x)
    n, c, h, w = shape
    y = torch.empty((n, 9 * c, h * w), device=DEV)
    args = H.im2col3_args(xd, y)
    ref = oracle.im2col3(x.numpy()).ravel()

    def check(what):
        torch.cuda.synchronize()
        assert H.hf_check_device_error() == 0
        assert np.array_equal(y.cpu().numpy().ravel(), ref), what
        y.fill_(-7.5)

    k = H.hf_register_kernel(H.IM2COL3)
    for threads in (32, 64, 96):
        for grid in (1, 5):
            H.hf_launch_single(k, args, threads, grid)
            check((threads, grid))
    for body in (H.BN_STATS, H.HIST256, H.UPSAMPLE2X, H.MAXPOOL3S2):
        ko = H.hf_register_kernel(body)
        oargs, keep = _other(body)
        for threads in (32, 64, 96):
            for cap in (0, 64, 96, 128):
                for first in (False, True):
                    f = H.hf_fuse(*((k, ko, threads) if first else (ko, k, 256 - threads)), 256, cap)
                    H.hf_launch(f, [args, oargs] if first else [oargs, args], 3)
                    check((body, threads, cap, first))
                    H.hf_destroy_fused(f)
        H.hf_destroy_kernel(ko)
    H.hf_destroy_kernel(k)


def test_lone_warp_takes_strips():
    """One warp an SM: rows of 64 columns cost strips 0.78 of what as many
    values cost the flat path, whose cost does not depend on the row."""
    k = H.hf_register_kernel(H.IM2COL3)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    best = []
    for side in (32, 64):
        x = torch.rand(1, (1 << 22) // side ** 2, side, side, device=DEV)
        y = torch.empty(1, 9 * x.shape[1], side * side, device=DEV)
        args = H.im2col3_args(x, y)
        times = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                H.hf_launch_single(k, args, 32, sms)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b))
        best.append(min(times[1:]))
    H.hf_destroy_kernel(k)
    assert best[1] < 0.9 * best[0]
