"""What is measured: forward inference of pattern- and connectivity-pruned 3x3 convolutions.

A case is one call that a program built on this library makes: a single layer through
``pp_conv_forward`` / ``pp_conv_forward_noalloc`` / ``pp_dense_forward``, or a whole network
through the executor (``runner.DeviceNet``), device-resident or from host buffers.  Packing,
upload and kernel choice belong to model loading and sit in ``prepare``, as in such a program.

Kinds of cases (``"kind"``):
  layer    one pruned layer.  ``"tune"``: the program calls ``pp_layer_autotune`` after loading;
           without it the library's default choice runs.  ``"entry"``: forward or noalloc.
  dense    one unpruned layer (all 9 taps).
  net      a network of ``"arch"`` vgg16 / style / sr.  ``"host"``: frames come from and go back
           to page-locked host memory (``pp_net_run_host``).
``"precision"`` is the library's own option for the tensor-core arithmetic: tf32x3 (its default)
or f16x3.  Flags: ``relu``, ``skip`` (a residual tensor is added), ``pool`` (2x2 max pool).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2004_11250_gb300 import ppconv as pp
from paper_2004_11250_gb300 import runner, synth

PRECISION = {"tf32x3": pp.PP_PRECISION_TF32X3, "f16x3": pp.PP_PRECISION_F16X3}


def _layer(name, N, Ci, Co, H, W, keep, P=8, ring=True, precision="tf32x3", tune=True, entry="forward", relu=True,
           skip=False, pool=False):
    c = dict(kind="layer", N=N, Ci=Ci, Co=Co, H=H, W=W, keep=keep, P=P, ring=ring, precision=precision, tune=tune,
             entry=entry, relu=relu, skip=skip, pool=pool)
    return dict(c, name=name) if name else c


def _dense(name, N, Ci, Co, H, W, relu=True, skip=False, pool=False):
    c = dict(kind="dense", N=N, Ci=Ci, Co=Co, H=H, W=W, relu=relu, skip=skip, pool=pool)
    return dict(c, name=name) if name else c


def _net(name, arch, H, W, precision="tf32x3", host=False, C=0, depth=0, keep=0.3):
    c = dict(kind="net", arch=arch, H=H, W=W, C=C, depth=depth, keep=keep, precision=precision, host=host)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest call: one 16 -> 16 layer on a 32 x 32 map.  Latency and the host side of a launch decide.
        _layer("single_16x32x32", 1, 16, 16, 32, 32, 0.5, relu=False),
        # The headline: a frame of the pruned VGG-16 trunk, batch 1, replayed on the device.
        _net("vgg16_224", "vgg16", 224, 224, keep=0.3),
        # The same trunk as a server runs it: frames arrive in and return to pinned host memory; fp16-split arithmetic.
        _net("vgg16_224_host_f16", "vgg16", 224, 224, precision="f16x3", host=True, keep=0.3),
        # Style transfer: the residual trunk of a 512 x 512 frame, five blocks of two 128 -> 128 layers.
        _net("style_128x128", "style", 128, 128, C=128, depth=5, keep=0.25),
        # Super resolution: one of the eighteen 64 -> 64 layers on a 720p frame, in both arithmetics.
        _layer("sr_layer_720p", 1, 64, 64, 720, 1280, 0.4),
        _layer("sr_layer_720p_f16", 1, 64, 64, 720, 1280, 0.4, precision="f16x3"),
        # The same layer on a photograph of odd size (rows not 16-byte aligned).
        _layer("sr_layer_321x481", 1, 64, 64, 321, 481, 0.4),
        # The stack's last layer, left dense: 64 -> 1 plus the residual image.
        _dense("sr_last_720p", 1, 64, 1, 720, 1280, relu=False, skip=True),
        # A layer that pruning left alone inside a network: dense 64 -> 64.
        _dense("dense_64_56x56", 1, 64, 64, 56, 56),
        # Batched throughput: 256 -> 256 at 56 x 56, batch 8, a seed-chosen set of 12 patterns, fp16 split.
        _layer("batch8_256_56x56_f16", 8, 256, 256, 56, 56, 0.35, P=12, ring=False, precision="f16x3", relu=False),
        # Odd channel counts and sizes with a residual, called as loaded, without tuning.
        _layer("odd_100_200_45x61", 3, 100, 200, 45, 61, 0.5, P=6, ring=False, tune=False, skip=True),
        # A late pooled layer inside a program that may not allocate: 512 -> 512 at 28 x 28, batch 1.
        _layer("noalloc_512_28x28_pool", 1, 512, 512, 28, 28, 0.3, tune=False, entry="noalloc", pool=True),
    ]


# ------------------------------------------------------------------ drawn cases


def _log(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case: layers of 8 .. 512 channels on maps of 7 .. 720 x 1280 pixels, dense layers of 1 .. 96 channels,
    and the three networks on other frame sizes.  Dense work (all 9 taps) stays below the 720p layer's."""
    kind = rng.choice(["layer", "layer", "layer", "layer", "dense", "net"])
    if kind == "net":
        arch = rng.choice(["vgg16", "style", "sr"])
        precision = rng.choice(["tf32x3", "f16x3"])
        host = rng.random() < 0.3
        if arch == "vgg16":
            return _net(None, arch, 32 * rng.randint(2, 7), 32 * rng.randint(2, 7), precision, host, keep=round(rng.uniform(0.2, 0.5), 2))
        if arch == "style":
            return _net(None, arch, rng.randint(32, 128), rng.randint(32, 128), precision, host, C=rng.choice([64, 96, 128]),
                        depth=rng.randint(1, 5), keep=round(rng.uniform(0.2, 0.5), 2))
        return _net(None, arch, _log(rng, 32, 360), _log(rng, 32, 360), precision, host, C=64, depth=rng.randint(2, 8),
                    keep=round(rng.uniform(0.2, 0.5), 2))
    flags = dict(relu=rng.random() < 0.7, skip=rng.random() < 0.25, pool=rng.random() < 0.2)
    most = 9.0 * 64 * 64 * 720 * 1280
    while True:
        if kind == "layer":
            Ci, Co = _log(rng, 8, 512), _log(rng, 8, 512)
            if rng.random() < 0.4:  # equal, round channel counts are the common ones
                Ci = Co = rng.choice([64, 128, 256, 512])
        else:
            Ci, Co = rng.choice([(rng.randint(1, 4), _log(rng, 16, 96)), (_log(rng, 16, 96), rng.randint(1, 4)),
                                 (_log(rng, 8, 96), _log(rng, 8, 96))])
        N = rng.choice([1, 1, 1, 2, 3, 4, 8])
        H, W = _log(rng, 7, 720), _log(rng, 7, 1280)
        if flags["pool"]:
            H, W = H + H % 2, W + W % 2
        macs = 9.0 * Ci * Co * N * H * W
        # a dense inner layer is an exception in a pruned network: small and middling ones
        if macs <= (most if kind == "layer" else most / 50 if min(Ci, Co) > 16 else most / 4):
            break
    if kind == "dense":
        return _dense(None, N, Ci, Co, H, W, **flags)
    entry = "noalloc" if Co > 64 and W <= 126 and rng.random() < 0.25 else "forward"
    if entry == "noalloc" and flags["pool"] and W > 118:  # the flat kernel pools row pairs of one tile
        entry = "forward"
    return _layer(None, N, Ci, Co, H, W, round(rng.uniform(0.2, 1.0), 2), rng.choice([4, 8, 12]), rng.random() < 0.5,
                  rng.choice(["tf32x3", "f16x3"]), rng.random() < 0.6 and entry == "forward", entry, **flags)


# ------------------------------------------------------------------ inputs (from the seed alone)


def _ring():
    ring = (0, 1, 2, 5, 8, 7, 6, 3)
    return [sorted({4, ring[s], ring[(s + 1) % 8], ring[(s + 2) % 8]}) for s in range(8)]


def _patterns(rng, P, ring):
    if ring:
        return np.array(_ring()[:P] if P <= 8 else _ring(), np.uint8)
    around = [(a, b, c) for a in range(9) for b in range(a + 1, 9) for c in range(b + 1, 9) if 4 not in (a, b, c)]
    pick = np.sort(rng.choice(len(around), size=P, replace=False))
    return np.array([sorted(around[i] + (4,)) for i in pick], np.uint8)


def _pruned(rng, Co, Ci, taps, keep, std, bias=True):
    """Weights of a pruned layer: uniform patterns, exactly round(keep Co Ci) kernels kept, normal values."""
    ids = rng.integers(0, len(taps), (Co, Ci)).astype(np.uint8)
    mask = np.zeros(Co * Ci, np.uint8)
    mask[rng.permutation(Co * Ci)[: max(1, int(keep * Co * Ci + 0.5))]] = 1
    mask = mask.reshape(Co, Ci)
    on = np.zeros((len(taps), 9), bool)
    for p, t in enumerate(taps):
        on[p, t] = True
    w = rng.standard_normal((Co, Ci, 9), np.float32) * np.float32(std)
    w[w == 0] = np.float32(std)
    w = np.where(on[ids] & (mask == 1)[:, :, None], w, np.float32(0))
    b = (rng.standard_normal(Co) * 0.01).astype(np.float32) if bias else None
    return synth.PrunedLayer(w, mask, ids, taps, b)


def _dense_weights(rng, Co, Ci):
    w = rng.standard_normal((Co, Ci, 9), np.float32) * np.float32(math.sqrt(2.0 / (9 * Ci)))
    return synth.DenseLayer(w, (rng.standard_normal(Co) * 0.01).astype(np.float32))


def _he(Ci):
    return math.sqrt(2.0 / (9 * Ci))


def _ops(case, rng):
    """(ops, input shape, input range) of a network."""
    taps, keep, ops = np.array(_ring(), np.uint8), case["keep"], []
    if case["arch"] == "vgg16":
        ci = 3
        for item in (64, 64, "P", 128, 128, "P", 256, 256, 256, "P", 512, 512, 512, "P", 512, 512, 512):
            if item == "P":
                ops[-1].pool = True
                continue
            ops.append(synth.Op(_pruned(rng, item, ci, taps, keep if ops else 1.0, 2.25 * _he(ci)), relu=True))
            ci = item
        return ops, (1, 3, case["H"], case["W"]), (0.0, 1.0)
    if case["arch"] == "style":
        C = case["C"]
        for _ in range(case["depth"]):
            at = len(ops)
            ops.append(synth.Op(_pruned(rng, C, C, taps, keep, 0.05, False), relu=True))
            ops.append(synth.Op(_pruned(rng, C, C, taps, keep, 0.05, False), skip_from=at))
        return ops, (1, C, case["H"], case["W"]), (-1.0, 1.0)
    C = case["C"]
    ops.append(synth.Op(_dense_weights(rng, C, 1), relu=True))
    for _ in range(case["depth"]):
        ops.append(synth.Op(_pruned(rng, C, C, taps, keep, 2.25 * _he(C)), relu=True))
    ops.append(synth.Op(_dense_weights(rng, 1, C), skip_from=0))
    return ops, (1, 1, case["H"], case["W"]), (0.0, 1.0)


def _uniform(seed, shape, lo, hi, device):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return torch.empty(shape, device=device, dtype=torch.float32).uniform_(lo, hi, generator=g)


def _inputs(case, seed):
    """(ops, x on the host for host networks and on the device otherwise, skip tensor or None)."""
    rng = np.random.default_rng([7, seed])
    if case["kind"] == "net":
        ops, shape, (lo, hi) = _ops(case, rng)
        return ops, _uniform(seed, shape, lo, hi, "cpu" if case["host"] else "cuda"), None
    N, Ci, Co, H, W = (case[k] for k in ("N", "Ci", "Co", "H", "W"))
    if case["kind"] == "dense":
        L = _dense_weights(rng, Co, Ci)
    else:
        L = _pruned(rng, Co, Ci, _patterns(rng, case["P"], case["ring"]), case["keep"], 0.05)
    op = synth.Op(L, relu=case["relu"], pool=case["pool"])
    x = _uniform(seed, (N, Ci, H, W), -1.0, 1.0, "cuda")
    skip = _uniform(seed + 1000003, (N, Co, H, W), -1.0, 1.0, "cuda") if case["skip"] else None
    return [op], x, skip


# ------------------------------------------------------------------ the calls


class _State:
    """What the program keeps between calls."""

    def __init__(self, case, seed):
        self.stream = torch.cuda.Stream()
        ops, self.x, self.skip = _inputs(case, seed)
        self.case, self.net, self.layer = case, None, None
        torch.cuda.synchronize()
        if case["kind"] == "net":
            # the executor's description carries the input's shape; the values are given to each run
            spec = synth.Net(case["arch"], np.empty(tuple(self.x.shape), np.float32), ops)
            self.net = runner.DeviceNet(spec, use_graph=True, stream=self.stream, precision=PRECISION[case["precision"]])
            if case["host"]:
                self.x = self.x.pin_memory()
                self.y = torch.empty(self.net.out_shape, dtype=torch.float32).pin_memory()
            else:
                self.y = torch.empty(self.net.out_shape, device="cuda")
        else:
            op = ops[0]
            precision = PRECISION[case.get("precision", "tf32x3")]
            self.layer = runner.DeviceLayer(op.layer, self.stream, precision=precision)
            N, _, H, W = self.x.shape
            self.flags = (pp.PP_RELU if op.relu else 0) | (pp.PP_ADD_SKIP if case["skip"] else 0) | (pp.PP_POOL2 if op.pool else 0)
            self.shape = (N, H, W)
            self.y = torch.empty((N, case["Co"], H // 2, W // 2) if op.pool else (N, case["Co"], H, W), device="cuda")
            if case.get("tune"):
                pp.pp_layer_autotune(self.layer.handle, N, H, W, self.flags, self.stream)
        torch.cuda.synchronize()

    def __del__(self):
        # the program's own teardown: handles go before the library does
        if getattr(self, "net", None) is not None:
            self.net.close()
        if getattr(self, "layer", None) is not None:
            self.layer.close()


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    if s.net is not None:
        if s.case["host"]:
            s.net.run_host(s.x, s.y, s.stream)
        else:
            s.net.run(s.x, s.y, s.stream)
        return s.y
    N, H, W = s.shape
    if s.case.get("entry") == "noalloc":
        pp.pp_conv_forward_noalloc(s.layer.handle, s.x, s.y, s.skip, N, H, W, s.flags, s.stream)
    else:
        s.layer.forward(s.x, s.y, s.skip, N, H, W, s.flags, s.stream)
    return s.y


# ------------------------------------------------------------------ what a pass cannot do without, and how exact it is


def _shapes(case):
    """(Ci, Co, H, W, kept taps, pool, skip) of every op, and N."""
    if case["kind"] != "net":
        n = case["Co"] * case["Ci"]
        taps = 9 * n if case["kind"] == "dense" else 4 * max(1, int(case["keep"] * n + 0.5))
        return [(case["Ci"], case["Co"], case["H"], case["W"], taps, case["pool"], case["skip"])], case["N"]
    out, H, W, keep = [], case["H"], case["W"], case["keep"]
    if case["arch"] == "vgg16":
        ci = 3
        for i, item in enumerate((64, -64, 128, -128, 256, 256, -256, 512, 512, -512, 512, 512, 512)):
            co, pool = abs(item), item < 0
            out.append((ci, co, H, W, 4 * max(1, int((keep if i else 1.0) * ci * co + 0.5)), pool, False))
            ci = co
            H, W = (H // 2, W // 2) if pool else (H, W)
        return out, 1
    C = case["C"]
    mid = 4 * max(1, int(keep * C * C + 0.5))
    if case["arch"] == "style":
        return [(C, C, H, W, mid, False, bool(i & 1)) for i in range(2 * case["depth"])], 1
    return [(1, C, H, W, 9 * C, False, False)] + [(C, C, H, W, mid, False, False)] * case["depth"] + [(C, 1, H, W, 9 * C, False, True)], 1


def work(case):
    """Surviving multiply-adds (2 FLOP each) of every op; the input and any residual read once, the output written
    once, each kept weight (and a dense layer's every weight) read once.  Activations between ops are the
    executor's own and not counted."""
    ops, N = _shapes(case)
    flops = sum(2.0 * N * H * W * t for _, _, H, W, t, _, _ in ops)
    Ci, _, H0, W0 = ops[0][:4]
    _, Co, H, W, _, pool, _ = ops[-1]
    out = N * Co * (H // 2 * (W // 2) if pool else H * W)
    size = N * Ci * H0 * W0 + out + sum(t for _, _, _, _, t, _, _ in ops)
    if case["kind"] != "net" and case["skip"]:
        size += N * Co * H * W
    return {"bytes": 4.0 * size, "flops": flops}


def tolerance(case):
    """Results in 32 bits.  The tensor cores' 32-bit sums of 9 Ci products (three per weight) measured, against 64
    bits, 2e-6 (64 channels) to 5e-6 (512) in tf32x3 and a fourth to two thirds of that in f16x3; plain 32-bit sums of
    the dense layers up to 4e-7.  Through a network the errors add up: 2.4e-5 over VGG-16's 13 layers in tf32x3, 5e-6
    in f16x3, up to 5e-6 in the residual networks.  About four times what was measured; single values stray up to
    ten times further."""
    f16 = case.get("precision") == "f16x3"
    if case["kind"] == "net":
        rel = (1e-4 if not f16 else 2e-5) if case["arch"] == "vgg16" else 2e-5
    elif case["kind"] == "dense":
        rel = 2e-6
    else:
        rel = (6e-6 + 3e-5 * case["Ci"] / 512) * (0.6 if f16 else 1.0)
    return {"rel": rel, "max": 10 * rel}


def _conv64(x, w):
    """3x3, zero padding 1, in 64 bits: one product of matrices per tap.  x [N][Ci][H][W], w [Co][Ci][9]."""
    N, Ci, H, W = x.shape
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
    y = torch.zeros((N, w.shape[0], H * W), dtype=torch.float64, device=x.device)
    for t in range(9):
        if bool((w[:, :, t] != 0).any()):
            s = xp[:, :, t // 3: t // 3 + H, t % 3: t % 3 + W].reshape(N, Ci, H * W)
            y += torch.matmul(w[:, :, t], s)
    return y.reshape(N, -1, H, W)


def exact(case, seed):
    ops, x, skip = _inputs(case, seed)
    acts = [x.cuda().double()]
    for op in ops:
        L = op.layer
        y = _conv64(acts[-1], torch.from_numpy(L.w).cuda().double())
        if L.bias is not None:
            y += torch.from_numpy(L.bias).cuda().double()[None, :, None, None]
        if skip is not None:
            y += skip.double()
        elif op.skip_from >= 0:
            y = y + acts[op.skip_from]
        if op.relu:
            y = torch.relu(y)
        if op.pool:
            y = torch.nn.functional.max_pool2d(y, 2)
        acts.append(y)
    return acts[-1].cpu() if case.get("host") else acts[-1]
