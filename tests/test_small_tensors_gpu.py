"""The resampling bodies' lines between small tensors (strips or a thread per
output) and the flat path: the same bits on both sides of each, values a
maximum must order included."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_util import DEV, single  # noqa: E402
from paper_2007_01277_gb300 import hfuse as H  # noqa: E402

ARGS = {H.UPSAMPLE2X: H.upsample2x_args, H.MAXPOOL3S2: H.maxpool3s2_args, H.IM2COL3: H.im2col3_args}


def _launch(body, x, threads, grid):
    n, c, h, w = x.shape
    size = {H.UPSAMPLE2X: 4 * x.numel(), H.IM2COL3: 9 * x.numel(),
            H.MAXPOOL3S2: n * c * ((h - 1) // 2 + 1) * ((w - 1) // 2 + 1)}[body]
    buf = torch.full((size + 8,), -7.5, device=DEV)
    shape = {H.UPSAMPLE2X: (n, c, 2 * h, 2 * w), H.IM2COL3: (n, 9 * c, h * w),
             H.MAXPOOL3S2: (n, c, (h - 1) // 2 + 1, (w - 1) // 2 + 1)}[body]
    y = buf[4: 4 + size].view(shape)
    single(body, ARGS[body](x, y), threads, grid)
    torch.cuda.synchronize()
    assert H.hf_check_device_error() == 0
    assert (buf[:4] == -7.5).all() and (buf[4 + size:] == -7.5).all()
    return buf[4: 4 + size].view(torch.int32)


@pytest.mark.parametrize("shape", [(1, 2, 1, 4), (3, 5, 12, 8), (2, 7, 9, 40), (1, 9, 20, 48), (2, 3, 24, 60),
                                   (1, 3, 11, 75), (2, 2, 7, 338), (1, 2, 5, 501), (1, 1, 3, 2049)])
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("body", list(ARGS))
def test_same_bits_whatever_the_grid(body, shape, off):
    g = torch.Generator().manual_seed(sum(shape))
    x = torch.randn(shape, generator=g)
    special = torch.tensor([float("nan"), float("inf"), -float("inf"), 0.0, -0.0])
    pick = torch.randint(0, 40, x.shape, generator=g)
    x = torch.where(pick < 5, special[pick.clamp(max=4)], x)
    xd = torch.empty(x.numel() + 1, device=DEV)[off: off + x.numel()].view(shape).copy_(x)
    ref = _launch(body, xd, 256, 0)
    for threads, grid in ((32, 1), (32, 2), (64, 2), (96, 3), (256, 1), (256, 9), (768, 5), (512, 152)):
        y = _launch(body, xd, threads, grid)
        nan = ref.view(torch.float32).isnan()
        assert torch.equal(y.view(torch.float32).isnan(), nan)
        assert torch.equal(y[~nan], ref[~nan])
