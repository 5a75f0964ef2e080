"""The measured cases: what programs that use this library have it do.

A kernel is written "body:sizes", as in "bn:8x64x32x32" (NCHW), "poly:1048576"
(elements) or "tmpl:16777216:16:2:8192" (floats, multiply-adds per 16 bytes,
barriers, staged bytes).  A case is one of

  pair    two kernels fused by hf_fuse and launched by hf_launch
  nway    several kernels in one persistent launch (hf_fuse_n, hf_launch)
  single  one kernel alone (hf_launch_single, or hf_bn_stats_noalloc)
  train   a run of the cost model's training kernel (hf_mlp_train)
  score   one scoring launch of the cost model (hf_mlp_forward)

Inputs follow the distributions of the library's workloads and are drawn on
the device from the seed.  The thread splits, register caps and blocks per SM
are those the library's own searches, tests and benchmark launch with; 0
blocks per SM leaves the grid to the library.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2007_01277_gb300 import hfuse as H

POLY_ITERS = 64
BF16_ALPHA = 0.5
TMPL_A, TMPL_B = 0.999, 0.001
HASH_TARGET, HASH_CAP = 1 << 16, 1024
HASH = {"sha256d": H.SHA256D, "blake256": H.BLAKE256, "blake2b": H.BLAKE2B}
IMAGE = ("bn", "bn_noalloc", "upsample", "maxpool", "im2col")
# 32-bit operations a nonce needs when it is hashed whole (rounds times
# operations per round; three-input adds and XORs counted once)
HASH_OPS = {"sha256d": 2752, "blake256": 1568, "blake2b": 2112}


def listed():
    return [
        # The smallest call: two kernels whose work is a few thousand values.
        # What counts is the launch and the host path before it.
        dict(name="tiny_pair", kind="pair", a="bn:2x8x16x12", b="poly:3000", split=256, d0=512, regcap=0, bps=0),
        # The paper's plain pair at the library's small size: statistics of
        # an activation tensor beside a multiply-add bound kernel.
        dict(name="bn_poly", kind="pair", a="bn:8x64x32x32", b="poly:1048576", split=256, d0=512, regcap=0, bps=0),
        # Two memory-bound image kernels at the library's large size, in the
        # launch shape that its search picks.
        dict(name="upsample_maxpool", kind="pair", a="upsample:32x64x128x128", b="maxpool:32x128x112x112", split=128,
             d0=512, regcap=0, bps=1),
        # A memory-bound kernel beside a generator, the library's largest
        # pair, in the launch shape that its search picks.
        dict(name="hist_philox", kind="pair", a="hist:268435456", b="philox:67108864", split=128, d0=256, regcap=64,
             bps=2),
        # Image kernels at odd sizes whose rows are not multiples of 16
        # bytes, as in networks with unpadded stems (75, 147).
        dict(name="resample_ragged", kind="pair", a="upsample:8x64x75x75", b="maxpool:8x64x147x147", split=256, d0=512,
             regcap=0, bps=0),
        # The late layers of a convolutional network: many channels of small
        # images (7x7, 14x14).
        dict(name="bn_im2col_deep", kind="pair", a="bn:64x512x7x7", b="im2col:32x256x14x14", split=256, d0=512,
             regcap=0, bps=0),
        # The early layers of one: im2col of wide images, launched alone.
        dict(name="im2col_wide", kind="single", a="im2col:8x64x112x112", threads=256),
        # Two kernels of the cost model's corpus: one bound by memory with
        # barriers and staging, one by its multiply-adds.
        dict(name="template_pair", kind="pair", a="tmpl:16777216:16:2:8192", b="tmpl:6000004:256:1:0", split=128,
             d0=256, regcap=0, bps=0),
        # Mining: two nonce scans fused that keep their hits only (an eighth
        # of the library's hash workload).
        dict(name="hash_mining", kind="pair", a="sha256d:2097152", b="blake2b:2752512", split=256, d0=512, regcap=0,
             bps=0),
        # The library's headline: eight uneven kernels in one persistent
        # launch, in a plan of its autotuner.
        dict(name="nway8", kind="nway",
             kernels="bn:64x256x56x56 im2col:32x64x56x56 maxpool:32x128x112x112 upsample:32x64x128x128 "
                     "hist:67108864 philox:16777216 poly:4194304 bf16:134217728",
             interval_of="1 3 2 1 3 2 0 1", threads="256 128 96 32", regcap=0, bps=0),
        # Training of the learned cost model: forward, backward and Adam (a
        # hundredth of a full training run).
        dict(name="mlp_train", kind="train", rows=16086, steps=200, batch=64),
        # Scoring every candidate of a corpus' held-out pairs.
        dict(name="mlp_score", kind="score", rows=16086),
    ]


# ------------------------------------------------------------------ draws
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _image(rng, body, most):
    """Images of 4 to 224 columns, odd ones among them, and a total of at most
    `most` values."""
    if rng.random() < 0.5:
        h = w = rng.choice((7, 14, 28, 32, 35, 56, 64, 75, 112, 128, 147, 150))
    else:
        h, w = _log(rng, 4, 224), _log(rng, 4, 224)
    c = rng.choice((3, 16, 64, 96, 128, 256, 512))
    n = max(1, _log(rng, 1 << 14, most) // (c * h * w))
    return "%s:%dx%dx%dx%d" % (body, n, c, h, w)


def _kernel(rng, body, most):
    """One kernel that reads and writes about 8 * most bytes or less."""
    if body in ("bn", "bn_noalloc"):
        return _image(rng, body, most)
    if body in ("upsample", "im2col"):
        return _image(rng, body, most // 4)
    if body == "maxpool":
        return _image(rng, body, most)
    if body == "hist":
        return "hist:%d" % _log(rng, 1 << 14, 4 * most)
    if body == "philox":
        return "philox:%d" % _log(rng, 1 << 12, most // 2)
    if body == "poly":
        return "poly:%d" % _log(rng, 1 << 11, min(most, 1 << 22))
    if body == "bf16":
        return "bf16:%d" % _log(rng, 1 << 12, 2 * most)
    if body == "tmpl":
        return "tmpl:%d:%d:%d:%d" % (_log(rng, 1 << 18, most) // 4 * 4,
                                     rng.choice((0, 1, 2, 4, 8, 16, 32, 64, 128, 256)), rng.randrange(5),
                                     rng.choice((0, 4096, 8192, 16384, 24576, 32768, 49152)))
    return "%s:%d%s" % (body, _log(rng, 1 << 12, 1 << 21), rng.choice(("", ":digests")))


def draw(rng: random.Random):
    kind = rng.choice(("pair", "pair", "pair", "pair", "single", "single", "nway", "train", "score"))
    most = 1 << 25
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 500, 80000), steps=_log(rng, 20, 200), batch=rng.choice((64, 64, 48, 33, 16)))
    if kind == "score":
        return dict(kind=kind, rows=_log(rng, 100, 80000))
    if kind == "single":
        body = rng.choice(("bn", "bn_noalloc", "upsample", "maxpool", "im2col", "hist", "philox", "poly", "bf16", "tmpl",
                           "sha256d", "blake256", "blake2b"))
        return dict(kind=kind, a=_kernel(rng, body, most), threads=rng.choice((128, 256, 512)))
    if kind == "nway":
        bodies = rng.sample(("bn", "im2col", "maxpool", "upsample", "hist", "philox", "poly", "bf16"), rng.randrange(3, 9))
        ks = " ".join(_kernel(rng, b, most // 2) for b in bodies)
        ni = min(len(bodies), rng.choice((3, 4, 8)))
        place = list(range(ni)) + [rng.randrange(ni) for _ in range(len(bodies) - ni)]
        warps = [1] * ni
        for _ in range(16 - ni):
            warps[rng.randrange(ni)] += 1
        return dict(kind=kind, kernels=ks, interval_of=" ".join(map(str, place)),
                    threads=" ".join(str(32 * w) for w in warps), regcap=0, bps=0)
    pairs = (("bn", "poly"), ("upsample", "maxpool"), ("hist", "philox"), ("tmpl", "tmpl"), ("bn", "hist"),
             ("bn", "maxpool"), ("bn", "upsample"), ("bn", "im2col"), ("hist", "maxpool"), ("hist", "upsample"),
             ("hist", "im2col"), ("upsample", "maxpool"), ("maxpool", "im2col"), ("upsample", "im2col"),
             ("sha256d", "blake256"), ("sha256d", "blake2b"), ("blake256", "blake2b"))
    a, b = rng.choice(pairs)
    d0 = rng.choice((256, 512))
    return dict(kind=kind, a=_kernel(rng, a, most), b=_kernel(rng, b, most), split=rng.choice((d0 // 4, d0 // 2, 3 * d0 // 4)),
                d0=d0, regcap=rng.choice((0, 0, 64)), bps=rng.choice((0, 1, 2)))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _normal(shape, g):
    return torch.randn(shape, generator=g, device="cuda")


def _uniform(shape, lo, hi, g):
    return torch.rand(shape, generator=g, device="cuda").mul_(hi - lo).add_(lo)


def _split(spec):
    body, sizes = spec.split(":", 1)
    if body in IMAGE:
        return body, tuple(int(v) for v in sizes.split("x"))
    parts = sizes.split(":")
    return body, tuple(p if p == "digests" else int(p) for p in parts)


def _inputs(spec, seed):
    """The kernel's input tensors and values, from the seed alone."""
    body, s = _split(spec)
    g = _gen(seed)
    if body in ("bn", "bn_noalloc", "maxpool", "im2col"):
        return (_normal(s, g),)
    if body == "upsample":
        return (_uniform(s, 0.0, 1.0, g),)
    if body == "hist":
        return (torch.randint(0, 256, (s[0],), generator=g, device="cuda", dtype=torch.uint8),)
    if body == "philox":
        return (int(seed) * 2654435761 % (1 << 61),)
    if body == "poly":
        coef = _uniform((33,), -0.1, 0.1, g)
        return _uniform((s[0],), -1.0, 1.0, g), coef
    if body == "bf16":
        return tuple(_uniform((s[0],), -1.0, 1.0, g).to(torch.bfloat16) for _ in range(2))
    if body == "tmpl":
        return (_uniform((s[0],), -1.0, 1.0, g),)
    return (bytes(torch.randint(0, 256, (80,), generator=g, device="cuda", dtype=torch.uint8).tolist()),)


class _Kernel:
    """One kernel of a case: its argument block, what a program clears before
    each launch, and its outputs."""

    def __init__(self, spec, seed):
        body, s = _split(spec)
        inp = _inputs(spec, seed)
        self.clear = self.hits = None
        if body in ("bn", "bn_noalloc"):
            x = inp[0]
            mean, var = torch.empty(s[1], device="cuda"), torch.empty(s[1], device="cuda")
            self.body, self.out = H.BN_STATS, [mean, var]
            self.noalloc = (x, mean, var) if body == "bn_noalloc" else None
            self.args = H.bn_stats_args(x, mean, var, H.bn_stats_workspace(x))
            return
        self.noalloc = None
        if body == "upsample":
            y = torch.empty(s[:2] + (2 * s[2], 2 * s[3]), device="cuda")
            self.body, self.out, self.args = H.UPSAMPLE2X, [y], H.upsample2x_args(inp[0], y)
        elif body == "maxpool":
            y = torch.empty(s[:2] + ((s[2] - 1) // 2 + 1, (s[3] - 1) // 2 + 1), device="cuda")
            self.body, self.out, self.args = H.MAXPOOL3S2, [y], H.maxpool3s2_args(inp[0], y)
        elif body == "im2col":
            y = torch.empty((s[0], s[1] * 9, s[2] * s[3]), device="cuda")
            self.body, self.out, self.args = H.IM2COL3, [y], H.im2col3_args(inp[0], y)
        elif body == "hist":
            self.clear = torch.zeros(256, dtype=torch.int32, device="cuda")
            self.body, self.out, self.args = H.HIST256, [self.clear], H.hist256_args(inp[0], self.clear)
        elif body == "philox":
            y = torch.empty((s[0], 4), dtype=torch.int32, device="cuda")
            self.body, self.out, self.args = H.PHILOX, [y], H.philox_args(y, inp[0])
        elif body == "poly":
            y = torch.empty_like(inp[0])
            self.body, self.out = H.POLY, [y]
            self.args = H.poly_args(inp[0], y, inp[1].tolist(), POLY_ITERS)
        elif body == "bf16":
            y = torch.empty_like(inp[0])
            self.body, self.out, self.args = H.BF16_AXPY, [y], H.bf16_axpy_args(inp[0], inp[1], y, BF16_ALPHA)
        elif body == "tmpl":
            y = torch.empty_like(inp[0])
            self.body, self.out = H.STREAM_TMPL, [y]
            self.args = H.stream_tmpl_args(inp[0], y, s[1], s[2], s[3], TMPL_A, TMPL_B)
        else:
            # a scan: every digest, or its hits alone (stored in any order,
            # so a program sorts them)
            self.body = HASH[body]
            self.clear = torch.zeros(1 + HASH_CAP, dtype=torch.int32, device="cuda")
            count, hits = self.clear[:1], self.clear[1:]
            digests = torch.empty((s[0], 32), dtype=torch.uint8, device="cuda") if len(s) > 1 else None
            self.hits = hits
            self.out = [count] if digests is None else [count, digests]
            self.args = H.hash_scan_args(inp[0], s[0], 0, HASH_TARGET, digests, hits, count)

    def outputs(self):
        return self.out + ([torch.sort(self.hits).values] if self.hits is not None else [])


def _specs(case):
    if case["kind"] == "nway":
        return case["kernels"].split()
    return [case[k] for k in ("a", "b") if k in case]


def _mlp_inputs(case, seed):
    g = _gen(seed)
    X = torch.rand((case["rows"], 24), generator=g, device="cuda")
    Y = X[:, :4].sum(1) - 2.0 + 0.3 * torch.sin(6 * X[:, 5])
    bound = [(24 * 64, math.sqrt(6.0 / 88)), (64, 0.05), (64 * 64, math.sqrt(6.0 / 128)), (64, 0.05),
             (64, math.sqrt(6.0 / 65)), (1, 0.05)]
    P = torch.cat([_uniform((n,), -b, b, g) for n, b in bound])
    idx = None
    if case["kind"] == "train":
        idx = torch.randint(0, case["rows"], (case["steps"] * case["batch"],), generator=g, device="cuda",
                            dtype=torch.int32)
    return X, Y, P, idx


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("train", "score"):
        X, Y, P, idx = _mlp_inputs(case, seed)
        return dict(case, X=X, Y=Y, P=P, idx=idx, y=torch.empty(case["rows"], device="cuda"))
    ks = [_Kernel(sp, 31 * seed + 7 * j) for j, sp in enumerate(_specs(case))]
    handles = [H.hf_register_kernel(k.body) for k in ks]
    state = dict(case, ks=ks, handles=handles, args=[k.args for k in ks])
    state["grid"] = case.get("bps", 0) * torch.cuda.get_device_properties(0).multi_processor_count
    if kind == "pair":
        state["f"] = H.hf_fuse(handles[0], handles[1], case["split"], case["d0"], case["regcap"])
    elif kind == "nway":
        state["f"] = H.hf_fuse_n(handles, [int(v) for v in case["interval_of"].split()],
                                 [int(v) for v in case["threads"].split()], case["regcap"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "score":
        H.hf_mlp_forward(state["P"], state["X"], state["y"])
        return [state["y"]]
    if kind == "train":
        P = state["P"].clone()
        M, V = torch.zeros_like(P), torch.zeros_like(P)
        loss = torch.empty(state["steps"], device="cuda")
        grad = torch.empty_like(P)
        H.hf_mlp_train(P, M, V, state["X"], state["Y"], state["idx"], state["steps"], state["batch"], loss_out=loss,
                       grad_out=grad)
        return [P, M, V, loss, grad]
    for k in state["ks"]:
        if k.clear is not None:
            k.clear.zero_()
    if kind == "single":
        k = state["ks"][0]
        if k.noalloc is not None:
            H.hf_bn_stats_noalloc(*k.noalloc, threads=state["threads"])
        else:
            H.hf_launch_single(state["handles"][0], k.args, state["threads"])
    else:
        H.hf_launch(state["f"], state["args"], state["grid"])
    return [o for k in state["ks"] for o in k.outputs()]


# ------------------------------------------------------------------ work
def _work(spec):
    """(bytes read and written once, operations) of one kernel."""
    body, s = _split(spec)
    if body in IMAGE:
        n = s[0] * s[1] * s[2] * s[3]
        if body in ("bn", "bn_noalloc"):
            return 4 * n + 8 * s[1], 4 * n
        if body == "upsample":
            return 20 * n, 4 * 6 * n
        if body == "maxpool":
            o = s[0] * s[1] * ((s[2] - 1) // 2 + 1) * ((s[3] - 1) // 2 + 1)
            return 4 * (n + o), 8 * o
        return 40 * n, 0
    n = s[0]
    if body == "hist":
        return n + 1024, n
    if body == "philox":
        return 16 * n, 40 * n
    if body == "poly":
        return 8 * n, 2 * 33 * POLY_ITERS * n
    if body == "bf16":
        return 6 * n, 2 * n
    if body == "tmpl":
        return 8 * n, 2 * s[1] * (n // 4)
    return (32 * n if len(s) > 1 else 0) + 4, HASH_OPS[body] * n


def work(case):
    if case["kind"] == "score":
        return {"bytes": 100 * case["rows"] + 4 * 5825, "flops": 2 * 5696 * case["rows"]}
    if case["kind"] == "train":
        # rows gathered once a step; parameters and moments in and out; a
        # forward pass and a backward pass of twice its products
        n = case["steps"] * case["batch"]
        return {"bytes": 104 * n + 4 * 5825 * 6, "flops": 2 * 3 * 5696 * n}
    w = [_work(sp) for sp in _specs(case)]
    return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}


# ------------------------------------------------------------------ 64 bits
def _exact(spec, seed):
    body, s = _split(spec)
    inp = _inputs(spec, seed)
    F = torch.nn.functional
    if body in ("bn", "bn_noalloc"):
        x = inp[0].double()
        return [x.mean((0, 2, 3)), x.var((0, 2, 3), unbiased=False)]
    if body == "upsample":
        return [F.interpolate(inp[0].double(), scale_factor=2, mode="bilinear", align_corners=False)]
    if body == "maxpool":
        return [F.max_pool2d(inp[0].double(), 3, 2, 1)]
    if body == "im2col":
        return [torch.cat([F.unfold(v.double(), 3, padding=1) for v in inp[0].split(4)])]
    if body == "poly":
        x, c = inp[0].double(), inp[1].double().tolist()
        acc = torch.zeros_like(x)
        for _ in range(POLY_ITERS):
            for v in reversed(c):
                acc.mul_(x).add_(v)
        return [acc]
    if body == "bf16":
        return [inp[0].double().mul_(BF16_ALPHA).add_(inp[1].double())]
    if body == "tmpl":
        v = inp[0].double().view(-1, 4)
        a, b = float(np.float32(TMPL_A)), float(np.float32(TMPL_B))
        for j in range(4):
            for _ in range(s[1] // 4 + (1 if j < s[1] % 4 else 0)):
                v[:, j].mul_(a).add_(b)
        return [v.reshape(-1)]
    return [None] * {"hist": 1, "philox": 1}.get(body, 2 + (len(s) > 1))


def _mlp(P, X):
    W1, b1, W2, b2, w3, b3 = (P[i:j] for i, j in zip((0, 1536, 1600, 5696, 5760, 5824), (1536, 1600, 5696, 5760, 5824, 5825)))
    h1 = (X @ W1.view(64, 24).T + b1).relu()
    h2 = (h1 @ W2.view(64, 64).T + b2).relu()
    return h1, h2, h2 @ w3 + b3


def exact(case, seed):
    if case["kind"] not in ("train", "score"):
        outs = [_exact(sp, 31 * seed + 7 * j) for j, sp in enumerate(_specs(case))]
        flat = [o for out in outs for o in out]
        return flat if any(o is not None for o in flat) else None   # integer kernels only: nothing to say
    X, Y, P, idx = _mlp_inputs(case, seed)
    X, Y, P = X.double(), Y.double(), P.double()
    if case["kind"] == "score":
        return [_mlp(P, X)[2]]
    lr, b1, b2, eps = (float(np.float32(v)) for v in (1e-3, 0.9, 0.999, 1e-8))
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    losses, first = [], None
    for t in range(1, case["steps"] + 1):
        rows = idx[(t - 1) * case["batch"]: t * case["batch"]].long()
        x = X[rows]
        h1, h2, y = _mlp(P, x)
        e = y - Y[rows]
        losses.append((e * e).mean())
        dy = 2 * e / case["batch"]
        d2 = dy[:, None] * P[5760:5824] * (h2 > 0)
        d1 = d2 @ P[1600:5696].view(64, 64) * (h1 > 0)
        g = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), h2.T @ dy, dy.sum()[None]])
        first = g if first is None else first
        M = b1 * M + (1 - b1) * g
        V = b2 * V + (1 - b2) * g * g
        P = P - lr * (M / (1 - b1 ** t)) / ((V / (1 - b2 ** t)).sqrt() + eps)
    return [P, M, V, torch.stack(losses), first]
