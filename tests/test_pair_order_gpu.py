"""A pair fused either way round is one kernel with its intervals exchanged:
the same shared memory (each kernel's own, its ring included) and blocks per
SM, and the same results."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_util import DEV, check_bn, check_upsample  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402
from paper_2007_01277_gb300 import workloads as W  # noqa: E402


def _kernels():
    x = {n: f((2, 3, 40, 56)) for n, f in (("up", W.upsample_input), ("pool", W.maxpool_input), ("bn", W.bn_input),
                                           ("col", W.im2col_input))}
    h = W.hist_input(40007)
    d = {n: t.to(DEV) for n, t in x.items()}
    yu, yp = torch.empty(2, 3, 80, 112, device=DEV), torch.empty(2, 3, 20, 28, device=DEV)
    yc, bins = torch.empty(2, 27, 2240, device=DEV), torch.zeros(256, dtype=torch.int32, device=DEV)
    m, v, ws = torch.empty(3, device=DEV), torch.empty(3, device=DEV), H.bn_stats_workspace(d["bn"])
    hd = h.to(DEV)
    keep = (d, hd, ws)

    def hist():
        assert np.array_equal(bins.cpu().numpy().view(np.uint32), oracle.hist256(h.numpy()))
        bins.zero_()

    return keep, {
        "up": (H.UPSAMPLE2X, H.upsample2x_args(d["up"], yu), lambda: check_upsample(x["up"], yu)),
        "pool": (H.MAXPOOL3S2, H.maxpool3s2_args(d["pool"], yp),
                 lambda: np.testing.assert_array_equal(yp.cpu().numpy(), oracle.maxpool3s2p1(x["pool"].numpy()))),
        "bn": (H.BN_STATS, H.bn_stats_args(d["bn"], m, v, ws), lambda: check_bn(x["bn"], m, v)),
        "col": (H.IM2COL3, H.im2col3_args(d["col"], yc),
                lambda: np.testing.assert_array_equal(
                    yc.cpu().numpy().ravel(), oracle.im2col3(x["col"].numpy()).ravel())),
        "hist": (H.HIST256, H.hist256_args(hd, bins), hist)}


@pytest.mark.parametrize("pair", [("bn", "col"), ("col", "pool"), ("col", "up"), ("up", "pool"), ("hist", "col"),
                                  ("hist", "pool"), ("bn", "hist")])
@pytest.mark.parametrize("low", [32, 96, 384])
def test_either_order(pair, low):
    keep, kernels = _kernels()
    info = []
    for names, split in ((pair, low), (pair[::-1], 512 - low)):
        (ba, aa, ca), (bb, ab, cb) = (kernels[n] for n in names)
        ka, kb = H.hf_register_kernel(ba), H.hf_register_kernel(bb)
        f = H.hf_fuse(ka, kb, split, 512, 0)
        q = H.hf_query(f, [aa, ab])
        info.append((q["smem_bytes"], q["blocks_per_sm"]))
        H.hf_launch(f, [aa, ab], 3)
        torch.cuda.synchronize()
        ca()
        cb()
        H.hf_destroy_fused(f)
        for k in (ka, kb):
            H.hf_destroy_kernel(k)
    assert info[0] == info[1]
    assert H.hf_check_device_error() == 0
