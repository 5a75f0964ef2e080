"""Launch plans found again in the per-thread table: more plans than it holds,
in two orders and from two threads, and a stream switched between launches."""
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


def test_more_plans_than_the_table_holds():
    x = W.hist_input(70001).to(DEV)
    ref = oracle.hist256(x.cpu().numpy())
    k = H.hf_register_kernel(H.HIST256)
    shapes = [(32 * t, g) for t in (1, 3, 8, 16) for g in (0, *range(1, 40))]
    failed = []

    def run(order):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for threads, grid in order:
                bins = torch.zeros(256, dtype=torch.int32, device=DEV)
                H.hf_launch_single(k, H.hist256_args(x, bins), threads, grid)
                if not np.array_equal(bins.cpu().numpy().view(np.uint32), ref):
                    failed.append((threads, grid))

    workers = [threading.Thread(target=run, args=(o,)) for o in (shapes + shapes, shapes[::-1] + shapes)]
    for w in workers:
        w.start()
    for w in workers:
        w.join()
    assert not failed and H.hf_check_device_error() == 0


def test_launches_follow_the_current_stream():
    # a launch that took another stream than the current one would run
    # before the copy it depends on, which waits behind a long kernel
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    src = W.hist_input(1 << 16).to(DEV)
    slow = torch.rand(1 << 22, device=DEV)
    out = torch.empty_like(slow)
    kp, kh = H.hf_register_kernel(H.POLY), H.hf_register_kernel(H.HIST256)
    torch.cuda.synchronize()
    for s in (a, b, a):
        x = torch.zeros_like(src)
        bins = torch.zeros(256, dtype=torch.int32, device=DEV)
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            H.hf_launch_single(kp, H.poly_args(slow, out, [0.01] * 33), 256)
            x.copy_(src)
            H.hf_launch_single(kh, H.hist256_args(x, bins), 128)
        s.synchronize()
        assert np.array_equal(bins.cpu().numpy().view(np.uint32), oracle.hist256(src.cpu().numpy()))
