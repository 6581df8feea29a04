"""The work this library is measured on: pruned convolutions, pruned matrix products, a whole pruned
network, and the steps that turn dense weights into packed layers, each through the public entry points.

A case is a dict of plain values.  ``op`` says which call (or chain of calls) it stands for:

  conv    one block-punched convolution, NHWC, as a serving loop calls it for every layer
  linear  one block-based pruned GEMM (a 1x1 convolution over the pixels, or an FC layer)
  stack   the forward pass of the ResNet-50-topology network of pruned layers
  pack    one-shot magnitude pruning of a convolution's weights to a layer-wide rate, then packing
  repack  the same for a GEMM's weights (rows and columns per block), then packing and unpacking again
"""
from __future__ import annotations

import math

import torch

import paper_2012_00596_b200 as npas
from paper_2012_00596_b200 import inputs
from paper_2012_00596_b200.resnet50 import Resnet50Stack

PATTERNS = "patterns"          # tap sets of the eight four-tap patterns, blocks of 1 x 1, a quarter of the kernels cut


def _conv(name=None, **kw):
    c = dict(op="conv", N=1, H=14, W=14, C=64, K=64, R=3, stride=1, pad=1, Mb=16, Nb=8, taps=3, rate=0.0, masks="random",
             dtype="bf16", out="same", bias=True, residual=False, relu=True)
    c.update(kw)
    return c if name is None else dict(c, name=name)


def _linear(name=None, **kw):
    c = dict(op="linear", M=1, I=512, O=512, Bo=64, Bi=64, rows=32, cols=32, dtype="bf16", out="same", bias=True, residual=False,
             relu=True)
    c.update(kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call of the library: a single small fp32 layer, launch latency and host time
        _conv("conv_f32_one_image", N=1, H=16, W=16, C=32, K=32, Mb=8, Nb=4, taps=3, dtype="f32", bias=False, relu=False),
        # a middle layer of the network for one image: online inference, where latency counts
        _conv("conv_one_image", N=1, H=14, W=14, C=256, K=256, Mb=16, Nb=8, taps=3),
        # the same layer for an ordinary batch
        _conv("conv_batch_32", N=32, H=14, W=14, C=256, K=256, Mb=16, Nb=8, taps=3),
        # the largest single call: the block-size sweep's layer at its 16x16 / 3-of-9 point (the benchmark's workload)
        _conv("conv_sweep_64", N=64, H=28, W=28, C=512, K=512, Mb=16, Nb=16, taps=3, bias=False, relu=False),
        # an irregular layer: odd batch and image, channel counts that no power of two divides, stride 2, a shortcut to
        # add, and masks pruned to a layer-wide rate, so that blocks keep different numbers of taps
        _conv("conv_ragged_strided", N=7, H=45, W=37, C=96, K=176, Mb=16, Nb=8, rate=2.5, taps=0, stride=2, residual=True),
        # a pruned layer of the 1x1 kind for an ordinary batch (64 images of 7x7 pixels)
        _linear("gemm_3136", M=3136, I=512, O=2048, rows=16, cols=16),
        # the classifier at the end of a network: a thousand outputs, blocks that tile them, few rows
        _linear("fc_1000", M=64, I=2048, O=1000, Bo=40, Bi=64, rows=20, cols=32, relu=False),
        # the fp32 path of the matrix product
        _linear("gemm_f32", M=392, I=512, O=512, dtype="f32"),
        # the whole network for one image and for the batch it is benchmarked with
        dict(op="stack", N=1, H=224, name="stack_1"),
        dict(op="stack", N=64, H=224, name="stack_64"),
        # preparing a candidate network's layer: prune to a rate, pack (done for every layer of every candidate)
        dict(op="pack", K=512, C=512, R=3, Mb=16, Nb=8, rate=2.5, w_in="f32", name="pack_conv_512"),
        # the same for a GEMM layer, and reading the packed layer back
        dict(op="repack", O=2048, I=512, Bo=64, Bi=64, rows=32, cols=32, w_in="f32", name="repack_gemm_2048"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dense_flops(c):
    P = (c["H"] + 2 * c["pad"] - c["R"]) // c["stride"] + 1
    Q = (c["W"] + 2 * c["pad"] - c["R"]) // c["stride"] + 1
    return 2.0 * c["N"] * P * Q * c["C"] * c["K"] * c["R"] * c["R"]


def draw(rng):
    kind = rng.choice(["conv"] * 5 + ["linear"] * 3 + ["stack"] * 2 + ["pack", "repack"])
    if kind == "conv":
        f32 = rng.random() < 0.2
        Mb, Nb = rng.choice([(8, 4), (4, 4), (8, 8)] if f32 else [(16, 8), (16, 8), (16, 16), (16, 16), (32, 32), (8, 8), (4, 4), (1, 1)])
        step_c, step_k = max(16, Nb), max(16, Mb)
        top = 96 if f32 else 512
        C, K = (max(s, _log(rng, s, top) // s * s) for s in (step_c, step_k))
        if not f32 and rng.random() < 0.4:                       # the widths networks mostly have
            C, K = (rng.choice([64, 128, 256, 512]) for _ in range(2))
        c = _conv(N=_log(rng, 1, 64), H=_log(rng, 5, 64), W=_log(rng, 5, 64), C=C, K=K, Mb=Mb, Nb=Nb, stride=rng.choice([1, 1, 1, 2]),
                  dtype="f32" if f32 else "bf16", bias=rng.random() < 0.8, residual=rng.random() < 0.25, relu=rng.random() < 0.7)
        if not f32 and rng.random() < 0.15:
            c["out"] = "f32"
        if Mb == 1:
            c.update(masks=PATTERNS, taps=0)
        elif rng.random() < 0.35:
            c.update(rate=rng.choice([2.0, 2.5, 3.0, 5.0, 7.0]), taps=0)
        else:
            c["taps"] = rng.choice([1, 2, 3, 3, 4, 5, 9])
        while _dense_flops(c) > (1e9 if f32 else 2.3e11):        # no more than the largest listed layer
            side = max("NHW", key=lambda k: c[k])
            c[side] = max(1 if side == "N" else 5, c[side] * 2 // 3)
        return c
    if kind == "linear":
        f32 = rng.random() < 0.3
        c = _linear(M=_log(rng, 1, 2000 if f32 else 50000), I=64 * _log(rng, 1, 8 if f32 else 32), O=64 * _log(rng, 1, 8 if f32 else 32),
                    dtype="f32" if f32 else "bf16", bias=rng.random() < 0.8, residual=rng.random() < 0.3, relu=rng.random() < 0.7)
        c["Bo"], c["Bi"] = rng.choice([(64, 64), (64, 64), (32, 32), (16, 64)])
        if rng.random() < 0.2:                                   # a classifier
            c.update(M=_log(rng, 1, 256), O=1000, Bo=rng.choice([8, 40]), Bi=64, relu=False)
        c["rows"] = max(1, int(c["Bo"] * rng.choice([0.25, 0.5, 0.75, 1.0])))
        c["cols"] = max(1, int(c["Bi"] * rng.choice([0.25, 0.5, 0.75, 1.0])))
        if not f32 and rng.random() < 0.15:
            c["out"] = "f32"
        while 2.0 * c["M"] * c["I"] * c["O"] > (2e9 if f32 else 5e10):
            c["M"] = max(1, c["M"] * 2 // 3)
            if c["M"] < 100:
                c["I"] = max(64, c["I"] // 128 * 64)
        return c
    if kind == "stack":
        return dict(op="stack", N=_log(rng, 1, 64), H=32 * rng.randint(2, 7))
    if kind == "pack":
        Mb, Nb = rng.choice([(16, 8), (16, 16), (32, 32), (8, 8), (8, 4)])
        return dict(op="pack", K=32 * _log(rng, 1, 16), C=32 * _log(rng, 1, 16), R=rng.choice([3, 3, 3, 5]), Mb=Mb, Nb=Nb,
                    rate=rng.choice([2.0, 2.5, 3.0, 5.0, 7.0, 10.0]), w_in=rng.choice(["f32", "bf16"]))
    Bo, Bi = rng.choice([(64, 64), (32, 32), (16, 64)])
    return dict(op="repack", O=64 * _log(rng, 1, 32), I=64 * _log(rng, 1, 32), Bo=Bo, Bi=Bi, rows=max(1, Bo // rng.choice([1, 2, 4])),
                cols=max(1, Bi // rng.choice([1, 2, 4])), w_in=rng.choice(["f32", "bf16"]))


# ---- what a program has in hand before the call ------------------------------------------------

_DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _subsets(g, shape, n, keep):
    """Random `keep`-of-`n` subsets as 64-bit sets, one per block."""
    pick = torch.rand((*shape, n), generator=g, device="cuda").argsort(dim=-1)[..., :keep]
    return torch.ones_like(pick).bitwise_left_shift_(pick).sum(dim=-1)


def _pattern_masks(g, K, C):
    lib = torch.tensor(inputs.PATTERN_LIBRARY, dtype=torch.int64, device="cuda")
    tm = lib[torch.randint(0, len(lib), (K, C), generator=g, device="cuda")]
    return tm.masked_fill_(torch.rand((K, C), generator=g, device="cuda") < 0.25, 0)


def _prepare_conv(c, g):
    dt, odt = _DT[c["dtype"]], _DT["f32" if c["out"] == "f32" else c["dtype"]]
    K, R, C, Mb, Nb = c["K"], c["R"], c["C"], c["Mb"], c["Nb"]
    x = torch.randn((c["N"], c["H"], c["W"], C), generator=g, device="cuda").relu_().to(dt)
    w = (torch.randn((K, R, R, C), generator=g, device="cuda") * 0.02).to(dt)
    if c["masks"] == PATTERNS:
        tm = _pattern_masks(g, K, C)
    elif c["rate"] > 0:
        tm = npas.prune_bp_magnitude_global(w, Mb, Nb, rate=c["rate"])
    else:
        tm = _subsets(g, (K // Mb, C // Nb), R * R, c["taps"])
    P, Q = ((v + 2 * c["pad"] - R) // c["stride"] + 1 for v in (c["H"], c["W"]))
    return dict(x=x, blob=npas.pack_bp(w, tm, Mb, Nb), ws=npas.workspace(), odt=odt,
                bias=torch.randn((K,), generator=g, device="cuda") * 0.1 if c["bias"] else None,
                res=torch.randn((c["N"], P, Q, K), generator=g, device="cuda").to(odt) if c["residual"] else None)


def _prepare_linear(c, g):
    dt, odt = _DT[c["dtype"]], _DT["f32" if c["out"] == "f32" else c["dtype"]]
    O, I, Bo, Bi = c["O"], c["I"], c["Bo"], c["Bi"]
    w = (torch.randn((O, I), generator=g, device="cuda") * 0.02).to(dt)
    blocks = (O // Bo, I // Bi)
    blob = npas.pack_bb(w, _subsets(g, blocks, Bo, c["rows"]), _subsets(g, blocks, Bi, c["cols"]), Bo, Bi)
    return dict(x=torch.randn((c["M"], I), generator=g, device="cuda").relu_().to(dt), blob=blob, ws=npas.workspace(), odt=odt,
                bias=torch.randn((O,), generator=g, device="cuda") * 0.1 if c["bias"] else None,
                res=torch.randn((c["M"], O), generator=g, device="cuda").to(odt) if c["residual"] else None)


def _stack_layers(H, g):
    """The layers of inputs.config4 (same shapes, masks and weight scales), drawn on the GPU."""
    layers = []
    for name, kind, cin, cout, h, s, relu, src, res in inputs.resnet50_topology(H):
        lay = inputs.StackLayer(name, kind, cin, cout, h, s, relu, src, res)
        if kind == "pw":
            blocks = (cout // 64, cin // 64)
            lay.row_keep, lay.col_keep = (npas.mask_to_numpy(_subsets(g, blocks, 64, 32)) for _ in range(2))
            w = torch.randn((cout, cin), generator=g, device="cuda") * (math.sqrt(4.0 / cin) * (0.5 if (res >= 0 or not relu) else 1.0))
        else:
            (Mb, Nb), R = inputs.STACK_BLOCKS[kind], 7 if kind == "stem" else 3
            keep = 49 if kind == "stem" else 3
            lay.tap_mask = npas.mask_to_numpy(_subsets(g, (cout // Mb, cin // Nb), R * R, keep))
            w = torch.randn((cout, R, R, cin), generator=g, device="cuda") * math.sqrt(2.0 / (cin * keep))
        lay.w = w.to(torch.bfloat16).float().cpu().numpy()
        lay.bias = (torch.randn((cout,), generator=g, device="cuda") * 0.01).cpu().numpy()
        layers.append(lay)
    return layers


def prepare(case, seed):
    g = _gen(seed)
    if case["op"] == "conv":
        s = _prepare_conv(case, g)
    elif case["op"] == "linear":
        s = _prepare_linear(case, g)
    elif case["op"] == "stack":
        s = dict(net=Resnet50Stack(_stack_layers(case["H"], g)),
                 x=torch.randn((case["N"], case["H"], case["H"], 3), generator=g, device="cuda").to(torch.bfloat16))
    elif case["op"] == "pack":
        s = dict(w=(torch.randn((case["K"], case["R"], case["R"], case["C"]), generator=g, device="cuda") * 0.02).to(_DT[case["w_in"]]))
    else:
        s = dict(w=(torch.randn((case["O"], case["I"]), generator=g, device="cuda") * 0.02).to(_DT[case["w_in"]]))
    s["case"] = case
    return s


def run(s):
    c = s["case"]
    if c["op"] == "conv":
        return npas.conv2d_bp(s["x"], s["blob"], s["bias"], s["res"], stride=c["stride"], pad=c["pad"], relu=c["relu"],
                              out_dtype=s["odt"], ws=s["ws"])
    if c["op"] == "linear":
        return npas.linear_bb(s["x"], s["blob"], s["bias"], s["res"], relu=c["relu"], out_dtype=s["odt"], ws=s["ws"])
    if c["op"] == "stack":
        return s["net"].forward(s["x"])
    if c["op"] == "pack":
        masks = npas.prune_bp_magnitude_global(s["w"], c["Mb"], c["Nb"], rate=c["rate"])
        return masks, npas.pack_bp(s["w"], masks, c["Mb"], c["Nb"], packed_dtype=torch.bfloat16).data
    rows, cols = npas.prune_bb_magnitude(s["w"], c["Bo"], c["Bi"], c["rows"], c["cols"])
    blob = npas.pack_bb(s["w"], rows, cols, c["Bo"], c["Bi"], packed_dtype=torch.bfloat16)
    return (rows, cols, blob.data, *npas.unpack_bb(blob))


# ---- what a pass cannot do without -------------------------------------------------------------

def _kept_blocks(c):
    """(kept (block, tap) pairs, blocks) of a convolution's weights."""
    blocks = (c["K"] // c["Mb"]) * (c["C"] // c["Nb"])
    taps = c["R"] * c["R"]
    if c.get("masks") == PATTERNS:
        return blocks * 3, blocks                                  # four taps in three kernels of four
    return (int(math.floor(blocks * taps / c["rate"] + 0.5)) if c["rate"] > 0 else blocks * c["taps"]), blocks


def work(case):
    c = case
    if c["op"] == "conv":
        es, eo = (4 if c["dtype"] == "f32" else 2), (4 if "f32" in (c["dtype"], c["out"]) else 2)
        P, Q = ((v + 2 * c["pad"] - c["R"]) // c["stride"] + 1 for v in (c["H"], c["W"]))
        pairs, blocks = _kept_blocks(c)
        y = c["N"] * P * Q * c["K"]
        return {"bytes": c["N"] * c["H"] * c["W"] * c["C"] * es + y * eo * (2 if c["residual"] else 1) + pairs * (c["Mb"] * c["Nb"] * es + 4) +
                blocks * 4 + (c["K"] * 4 if c["bias"] else 0), "flops": 2.0 * c["N"] * P * Q * pairs * c["Mb"] * c["Nb"]}
    if c["op"] == "linear":
        es, eo = (4 if c["dtype"] == "f32" else 2), (4 if "f32" in (c["dtype"], c["out"]) else 2)
        blocks = (c["O"] // c["Bo"]) * (c["I"] // c["Bi"])
        kept = blocks * c["rows"] * c["cols"]
        return {"bytes": c["M"] * c["I"] * es + c["M"] * c["O"] * eo * (2 if c["residual"] else 1) + kept * es +
                blocks * (c["Bo"] + c["Bi"] + 6) + (c["O"] * 4 if c["bias"] else 0), "flops": 2.0 * c["M"] * kept}
    if c["op"] == "stack":
        n_bytes, flops = c["N"] * c["H"] * c["H"] * 6 + c["N"] * (c["H"] // 32) ** 2 * 2048 * 2, 0.0
        for _, kind, cin, cout, h, s, _, _, _ in inputs.resnet50_topology(c["H"]):
            px = ((h - 1) // s + 1) ** 2
            kept = cout * cin // 4 if kind == "pw" else cout * cin * (49 if kind == "stem" else 3)
            idx = (cout // 64) * (cin // 64) * 134 if kind == "pw" else kept // 32 + cout * cin // 32
            n_bytes += kept * 2 + idx + cout * 4
            flops += 2.0 * c["N"] * px * kept
        return {"bytes": n_bytes, "flops": flops}
    if c["op"] == "pack":
        n, es = c["K"] * c["C"] * c["R"] * c["R"], 4 if c["w_in"] == "f32" else 2
        pairs, blocks = _kept_blocks(c)
        copies = 2 if c["Mb"] % 16 == 0 and c["Nb"] % 16 == 0 and c["R"] == 3 else 1      # kept weights once, or again as tiles
        return {"bytes": n * es + n * 2 + pairs * (c["Mb"] * c["Nb"] * 2 * copies + 4) + blocks * 12, "flops": 2.0 * n}
    n, es = c["O"] * c["I"], 4 if c["w_in"] == "f32" else 2
    blocks = (c["O"] // c["Bo"]) * (c["I"] // c["Bi"])
    kept, tile = blocks * c["rows"] * c["cols"], blocks * c["Bo"] * max(16, (c["cols"] + 15) // 16 * 16)
    # weights in; the packed layer (dense image, kept values, tiles, lists) out; the dense weights and masks back out
    return {"bytes": n * es + n * 2 + kept * 2 + tile * 2 + blocks * (c["Bo"] + c["Bi"] + 6) + n * 2 + blocks * 32, "flops": 4.0 * n}


def tolerance(case):
    if case["op"] in ("pack", "repack"):
        return "exact"                     # masks are decided on fp64 sums in a fixed order, packing rounds once: same bits
    if case["op"] == "stack":
        return {"rel": 1e-2, "max": 0.1}   # bf16 activations through 53 layers: single roundings fall differently and carry on
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 1e-5}  # fp64 sums of fp32 products, one rounding
    if case["out"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}  # fp32 sums in another order
    return {"rel": 3e-3, "max": 1.6e-2}    # fp32 sums, one rounding to bf16
