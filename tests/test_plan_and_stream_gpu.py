"""The launch plans a thread finds again are those a thread that has none
makes; and a launch without a stream goes to the current one."""
import threading

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


def _fresh(fn):
    """fn() on a thread of its own, whose table is empty."""
    out = []
    t = threading.Thread(target=lambda: (torch.cuda.set_device(0), out.append(fn())))
    t.start()
    t.join()
    return out[0]


def test_plans_equal_those_of_a_fresh_thread():
    """More configurations than the table holds, those of one kernel differing
    in one number of the key at a time: ring kind (aligned input or not), staged
    bytes, block, split, intervals; in two orders, so that entries are replaced
    and found again."""
    buf = torch.rand(4 * 64 * 60 + 8, device=DEV)
    y = torch.empty(4 * 64 * 60 * 9, device=DEV)
    xs = [buf[o: o + 4 * 64 * 60].view(1, 4, 64, 60) for o in (0, 1)]
    up = [H.upsample2x_args(x, y[: 4 * x.numel()].view(1, 4, 128, 120)) for x in xs]
    col = [H.im2col3_args(x, y.view(1, 36, 64 * 60)) for x in xs]
    tm = [H.stream_tmpl_args(buf[:4096], y[:4096], 4, 1, sm, 0.9, 0.1) for sm in (0, 4096, 8192, 49152)]
    bins, hb = torch.zeros(256, dtype=torch.int32, device=DEV), W.hist_input(70001).to(DEV)
    hist = [H.hist256_args(hb[o:], bins) for o in (0, 1)]
    ku, kc, kt, kh = (H.hf_register_kernel(b) for b in (H.UPSAMPLE2X, H.IM2COL3, H.STREAM_TMPL, H.HIST256))
    queries = []
    for t in (32, 64, 128, 256, 512):
        for k, args in ((ku, up), (kc, col), (kt, tm), (kh, hist)):
            queries += [(lambda k=k, a=a, t=t: H.hf_query_single(k, a, t)) for a in args]
    fused = []
    for split in (32, 128, 224):
        for ka, kb, aa, ab in ((ku, kc, up, col), (kh, ku, hist, up), (kt, kt, tm, tm[::-1])):
            fused.append(H.hf_fuse(ka, kb, split, 256, 0))
            queries += [(lambda f=fused[-1], p=(p, q): H.hf_query(f, list(p))) for p in aa for q in ab]
    for io, it in (([0, 1, 2], [64, 64, 64]), ([0, 1, 2], [32, 64, 96]), ([0, 1, 1], [64, 128])):
        fused.append(H.hf_fuse_n([ku, kh, kc], io, it, 0))
        queries += [(lambda f=fused[-1], p=(p, q, r): H.hf_query(f, list(p))) for p in up for q in hist for r in col]
    assert len(queries) > 128
    here = [q() for q in queries]
    assert [q() for q in queries[::-1]] == here[::-1] and [q() for q in queries] == here
    for q, a in zip(queries, here):
        assert _fresh(q) == a
    for f in fused:
        H.hf_destroy_fused(f)
    for k in (ku, kc, kt, kh):
        H.hf_destroy_kernel(k)


def test_plans_keep_the_grid_apart():
    """One block and the whole device in turn, both plans in the table: the
    block takes the time of one."""
    x = torch.rand(1 << 18, device=DEV)
    args = H.poly_args(x, torch.empty_like(x), [0.01] * 33)
    k = H.hf_register_kernel(H.POLY)
    best = {1: 1e9, 0: 1e9}
    for _ in range(4):
        for grid in (1, 0):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            H.hf_launch_single(k, args, 256, grid)
            b.record()
            b.synchronize()
            best[grid] = min(best[grid], a.elapsed_time(b))
    H.hf_destroy_kernel(k)
    assert best[1] > 10 * best[0]


def test_launch_without_a_stream_takes_the_current_one():
    """The copy that the histogram depends on waits behind torch operations on
    the same stream; a launch on any other stream would run before it."""
    src = W.hist_input(1 << 16).to(DEV)
    ref = oracle.hist256(src.cpu().numpy())
    slow = torch.rand(1 << 26, device=DEV)
    k = H.hf_register_kernel(H.HIST256)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    x, bins = torch.zeros_like(src), torch.zeros(256, dtype=torch.int32, device=DEV)
    H.hf_launch_single(k, H.hist256_args(x, bins), 128)   # the plan is made, the binding initialised
    for s in (a, b, a, torch.cuda.default_stream()):
        x.zero_()
        bins.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            assert H._current_stream() == s.cuda_stream
            for _ in range(20):
                slow.mul_(1.0001)
            x.copy_(src)
            H.hf_launch_single(k, H.hist256_args(x, bins), 128)
            assert not s.query()   # the operations before the copy still run
        torch.cuda.synchronize()
        assert np.array_equal(bins.cpu().numpy().view(np.uint32), ref)
    H.hf_destroy_kernel(k)
