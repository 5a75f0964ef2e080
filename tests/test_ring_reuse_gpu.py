"""Kernels that follow one another on one interval's shared memory, each on a
bulk-copy ring over the bytes that the one before patched, counted or staged
in: totals that are not multiples of four, then rings of every kind."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import DEV, check_bf16, check_bn, check_upsample  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402
from paper_2007_01277_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("warps", [1, 4])
@pytest.mark.parametrize("grid", [1, 5])
def test_rings_one_after_another(warps, grid):
    xu, xm, xi = W.upsample_input((1, 1, 41, 15)), W.maxpool_input((3, 1, 35, 75)), W.maxpool_input((1, 3, 9, 7))
    xb, xh = W.bn_input((2, 3, 64, 32)), W.hist_input(50001)
    bx, by = W.bf16_inputs(40003)
    yu, ym = torch.empty(1, 1, 82, 30, device=DEV), torch.empty(3, 1, 18, 38, device=DEV)
    yi = torch.empty(1, 27, 63, device=DEV)
    mean, var = torch.empty(3, device=DEV), torch.empty(3, device=DEV)
    bins = torch.zeros(256, dtype=torch.int32, device=DEV)
    d = {n: t.to(DEV) for n, t in dict(u=xu, m=xm, i=xi, b=xb, h=xh, bx=bx, by=by).items()}
    out = torch.empty_like(d["bx"])
    ws = H.bn_stats_workspace(d["b"])
    sched = [(H.MAXPOOL3S2, H.maxpool3s2_args(d["m"], ym)), (H.IM2COL3, H.im2col3_args(d["i"], yi)),
             (H.UPSAMPLE2X, H.upsample2x_args(d["u"], yu)), (H.BN_STATS, H.bn_stats_args(d["b"], mean, var, ws)),
             (H.HIST256, H.hist256_args(d["h"], bins)), (H.BF16_AXPY, H.bf16_axpy_args(d["bx"], d["by"], out, 0.5))]
    for order in (sched, sched[::-1], sched[2:] + sched[:2]):
        bins.zero_()
        for t in (yu, ym, yi, out):
            t.fill_(-7.5)
        ks = [H.hf_register_kernel(b) for b, _ in order]
        f = H.hf_fuse_n(ks, [0] * len(ks), [32 * warps], 0)
        H.hf_launch(f, [a for _, a in order], grid)
        torch.cuda.synchronize()
        assert H.hf_check_device_error() == 0
        check_upsample(xu, yu)
        assert np.array_equal(ym.cpu().numpy(), oracle.maxpool3s2p1(xm.numpy()))
        assert np.array_equal(yi.cpu().numpy(), oracle.im2col3(xi.numpy()).reshape(1, 27, 63))
        check_bn(xb, mean, var)
        assert np.array_equal(bins.cpu().numpy().view(np.uint32), oracle.hist256(xh.numpy()))
        check_bf16(bx, by, out)
        H.hf_destroy_fused(f)
        for k in ks:
            H.hf_destroy_kernel(k)
