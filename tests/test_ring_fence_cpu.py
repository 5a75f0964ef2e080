"""A bulk-copy ring starts on shared memory that an earlier kernel of the same
N-way interval used with ordinary accesses (counters, staged values, values
patched into a stage).  Bulk copies go through another proxy, so a barrier
alone does not order them after those accesses: the ring's start has to issue
the proxy fence.  Shown on the source, since no run can show an order that
happened to hold."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_2007_01277_gb300", "csrc", "hf_device.cuh")


def _body(text, head):
    at = text.index("{", text.index(head))
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return re.sub(r"//[^\n]*", "", text[at: i + 1])
    raise AssertionError(head)


def test_ring_start_orders_earlier_accesses():
    text = open(SOURCE).read()
    ring = _body(text, "struct WarpRing")
    assert "fence.proxy.async.shared::cta" in _body(ring, "void refill_fence()")
    init = _body(ring, "void init(")
    assert "refill_fence();" in init[init.rindex("mbarrier"):]
