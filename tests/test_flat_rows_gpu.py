"""The flat path of the resampling bodies (rows of any length): every row
length at which its stage, its items or its store width change, planes
shorter and longer than an item, unaligned tensors (an unaligned input takes
no ring), and values a maximum must order."""
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

# 338 columns are the longest row of which three fit a 4 KB stage; 252 the
# longest of which four do; 169 and 170 where four odd rows no longer fit
SHAPES = [(3, 2, 7, 7), (5, 3, 1, 1), (2, 1, 3, 2), (1, 1, 1, 3), (40, 1, 2, 5), (2, 2, 14, 14), (3, 1, 75, 75),
          (1, 2, 30, 60), (2, 1, 9, 169), (2, 1, 8, 170), (1, 1, 7, 252), (1, 1, 6, 256), (1, 2, 5, 338),
          (1, 1, 5, 339), (1, 1, 4, 1015), (1, 1, 1500, 3), (300, 1, 1, 4), (1, 1, 1, 1021)]
LAUNCHES = [(32, 1), (64, 3), (256, 0), (768, 2)]


def out_like(body, shape):
    n, c, h, w = shape
    s = {H.UPSAMPLE2X: (n, c, 2 * h, 2 * w), H.MAXPOOL3S2: (n, c, (h - 1) // 2 + 1, (w - 1) // 2 + 1),
         H.IM2COL3: (n, 9 * c, h * w)}[body]
    return s


def launch(body, x, off_in, off_out, threads, grid):
    """One launch on views that start `off` floats into their buffers; the
    output with guard values around it, which must survive."""
    xd = torch.empty(x.numel() + 8, device=DEV)[off_in: off_in + x.numel()].view(x.shape)
    xd.copy_(x)
    so = out_like(body, x.shape)
    n = int(np.prod(so))
    buf = torch.full((n + 16,), -7.5, device=DEV)
    y = buf[8 + off_out: 8 + off_out + n].view(so)
    args = {H.UPSAMPLE2X: H.upsample2x_args, H.MAXPOOL3S2: H.maxpool3s2_args, H.IM2COL3: H.im2col3_args}[body](xd, y)
    single(body, args, threads, grid)
    torch.cuda.synchronize()
    assert H.hf_check_device_error() == 0
    assert (buf[: 8 + off_out] == -7.5).all() and (buf[8 + off_out + n:] == -7.5).all()
    return y


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("off_in,off_out", [(0, 0), (1, 0), (0, 1), (0, 2)])
def test_flat_rows(shape, off_in, off_out):
    x = W.upsample_input(shape, seed=sum(shape))
    z = W.maxpool_input(shape, seed=sum(shape))
    pool, col = oracle.maxpool3s2p1(z.numpy()), oracle.im2col3(z.numpy())
    for threads, grid in LAUNCHES:
        check_upsample(x, launch(H.UPSAMPLE2X, x, off_in, off_out, threads, grid))
        assert np.array_equal(launch(H.MAXPOOL3S2, z, off_in, off_out, threads, grid).cpu().numpy(), pool)
        assert np.array_equal(launch(H.IM2COL3, z, off_in, off_out, threads, grid).cpu().numpy(), col)


def _max(u, v):
    return np.where(v > u, v, u)


@pytest.mark.parametrize("w", [56, 75, 64])
def test_maxpool_orders_special_values(w):
    """Infinities, NaN and both zeros: 16-byte rows take each row's maximum
    from its left column on (a NaN there stays), other rows one running
    maximum that no NaN enters; equal values keep the first."""
    g = torch.Generator().manual_seed(w)
    x = torch.randn(2, 3, 21, w, generator=g)
    special = torch.tensor([float("nan"), float("inf"), -float("inf"), 0.0, -0.0])
    pick = torch.randint(0, 12, x.shape, generator=g)
    x = torch.where(pick < 5, special[pick.clamp(max=4)], x)
    p = np.pad(x.numpy(), ((0, 0), (0, 0), (1, 1), (1, 1)), constant_values=-np.inf)
    ho, wo = 11, (w - 1) // 2 + 1
    rows = []
    for ky in range(3):
        cols = [p[:, :, ky: ky + 2 * ho: 2, kx: kx + 2 * wo: 2][:, :, :ho, :wo] for kx in range(3)]
        left = cols[0] if w % 4 == 0 else _max(np.float32(-np.inf), cols[0])
        rows.append(_max(_max(left, cols[1]), cols[2]))
    ref = _max(_max(rows[0], rows[1]), rows[2])
    for threads, grid in LAUNCHES:
        y = launch(H.MAXPOOL3S2, x, 0, 0, threads, grid).cpu().numpy()
        assert np.array_equal(y.view(np.uint32)[~np.isnan(ref)], ref.view(np.uint32)[~np.isnan(ref)])
        assert np.array_equal(np.isnan(y), np.isnan(ref))
