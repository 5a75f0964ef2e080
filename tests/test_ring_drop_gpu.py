"""Which interval of a pair gives up its ring where shared memory does not hold
both: the larger one, but where a flat path would lose by it the one with fewer
bytes a warp."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402

RING = 2 * (4096 + 8)   # bytes of a warp's item ring


def _pool(w):
    x = torch.rand(2, 2, 19, w, device=DEV)
    y = torch.empty(2, 2, 10, (w - 1) // 2 + 1, device=DEV)
    return H.MAXPOOL3S2, H.maxpool3s2_args(x, y), (x, y)


def _up(w):
    x = torch.rand(2, 2, 19, w, device=DEV)
    y = torch.empty(2, 2, 38, 2 * w, device=DEV)
    return H.UPSAMPLE2X, H.upsample2x_args(x, y), (x, y)


# (upsample's columns, max pool's columns, their threads, warps that keep a ring)
@pytest.mark.parametrize("wu,wp,tu,tp,keep", [(15, 6, 128, 384, 4), (6, 15, 384, 128, 4), (15, 112, 128, 384, 4),
                                              (112, 6, 384, 128, 12), (75, 6, 384, 128, 12), (2, 250, 128, 384, 12),
                                              (112, 112, 128, 384, 4)])
def test_which_ring_goes(wu, wp, tu, tp, keep):
    """512 threads capped at 64 registers: two blocks an SM, each with room for
    12 of its 16 warps' rings."""
    (bu, au, ku), (bp, ap, kp) = _up(wu), _pool(wp)
    for first, second in (((bu, au, tu), (bp, ap, tp)), ((bp, ap, tp), (bu, au, tu))):
        ka, kb = H.hf_register_kernel(first[0]), H.hf_register_kernel(second[0])
        f = H.hf_fuse(ka, kb, first[2], 512, 64)
        q = H.hf_query(f, [first[1], second[1]])
        assert q["blocks_per_sm"] == 2
        assert keep * RING <= q["smem_bytes"] < keep * RING + 1024
        H.hf_destroy_fused(f)
        for k in (ka, kb):
            H.hf_destroy_kernel(k)
