"""The work that is measured: what a user of this package has it do, at the sizes of the
package's own configurations and at drawn sizes of the same ranges.

A case is a dict of plain values; its "kind" says which calls it makes:

conv        one integer convolution (``aqd.conv_int``), codes in, codes out
bottleneck  a 1x1 / 3x3 / 1x1 residual bottleneck, its layers chained
down_block  a stage-entry basic block: 3x3 stride 2, 1x1 stride 2 (int32), 3x3 with that skip
head        the shared detector head over its pyramid levels: the tower, then the output conv
head_layer  one tower layer over all levels (``aqd.conv_int_grouped``)
detector    a whole integer detector (``detector.IntDetector.forward``)
eltwise     the stand-alone requant and integer skip adds of an int32 tensor
codes       int32 codes packed, max-pooled and unpacked again
fake_quant  a training quantizer with a learnable interval, forward and backward
bn_stats    the per-level batch statistics of the multi-level batch norm

Every integer result is exact; the float32 training steps have the tolerance of their type.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2007_06919_gb300 import aqd, synth
from paper_2007_06919_gb300.detector import IntDetector

DEV = "cuda"


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # a first small layer: one 3x3 conv of a 32x32 map, where a call's latency is all there is
        dict(name="conv_small_2bit", kind="conv", n=1, h=32, w=32, cin=64, cout=64, k=3, stride=1, bits=2),
        # channel and spatial sizes that fit no tile, 3-bit codes, an input width of 96 channels
        dict(name="conv_ragged_3bit", kind="conv", n=2, h=67, w=101, cin=96, cout=160, k=3, stride=1, bits=3),
        # ResNet-50's C3 bottleneck at the size an 800-pixel image gives it
        dict(name="bottleneck_4bit_b2", kind="bottleneck", n=2, h=100, w=152, wide=512, mid=128, bits=4),
        # ResNet-18's third stage begins: stride-2 convs and an int32 downsample skip
        dict(name="down_block_4bit_b8", kind="down_block", n=8, h=100, w=168, cin=128, cout=256, bits=4),
        # the RetinaNet head of two 800x1333 images at 2 bits, all five pyramid levels
        dict(name="head_2bit_b2", kind="head", n=2, h=100, w=168, layers=4, bits=2),
        # one layer of that head at batch 16 and 8 bits
        dict(name="head_layer_8bit_b16", kind="head_layer", n=16, h=100, w=168, bits=8),
        # one image through the whole detector: serving at the lowest latency
        dict(name="detector_b1", kind="detector", n=1, h=800, w=1333, w_pad=1344),
        # a batch of eight: serving for throughput
        dict(name="detector_b8", kind="detector", n=8, h=800, w=1333, w_pad=1344),
        # int32 accumulators of a P3 level turned into codes: alone, with a skip, with an upsampled skip
        dict(name="eltwise_4bit_b8", kind="eltwise", n=8, h=100, w=168, c=256, bits=4, skip_bits=4),
        # a stem-sized map of codes: packed, pooled 3x3 stride 2, unpacked
        dict(name="codes_4bit_b8", kind="codes", n=8, h=400, w=672, c=64, bits=4),
        # an activation quantizer of the training step over a P3 level at batch 16
        dict(name="fake_quant_act_4bit", kind="fake_quant", numel=16 * 100 * 168 * 256, bits=4, weight=False),
        # the head's batch statistics over five levels at batch 16
        dict(name="bn_stats_b16", kind="bn_stats", n=16, h=100, w=168, c=256, levels=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "bottleneck", "down_block", "head", "head_layer", "detector",
                       "eltwise", "codes", "fake_quant", "bn_stats"])
    if kind == "conv":
        # any layer of a network: spatial sizes 7 to 200, 32 to 512 channels, strides 1 and 2
        k, stride = rng.choice([(1, 1), (3, 1), (3, 1), (3, 2), (1, 2)])
        return dict(kind=kind, n=_log(rng, 1, 8), h=_log(rng, 7, 120), w=_log(rng, 7, 200),
                    cin=32 * rng.choice([1, 2, 3, 4, 6, 8, 16]), cout=32 * rng.choice([1, 2, 3, 5, 8, 12, 16]),
                    k=k, stride=stride, bits=rng.choice([2, 3, 4]))
    if kind == "bottleneck":
        mid = rng.choice([64, 128, 256])
        return dict(kind=kind, n=rng.randint(1, 4), h=_log(rng, 13, 200), w=_log(rng, 13, 200), wide=4 * mid, mid=mid,
                    bits=rng.choice([2, 3, 4]))
    if kind == "down_block":
        cin = rng.choice([64, 128, 256])
        return dict(kind=kind, n=rng.randint(1, 8), h=_log(rng, 15, 120), w=_log(rng, 15, 180), cin=cin, cout=2 * cin,
                    bits=rng.choice([2, 3, 4]))
    if kind == "head":
        return dict(kind=kind, n=_log(rng, 1, 8), h=_log(rng, 16, 120), w=_log(rng, 16, 180), layers=rng.randint(1, 4),
                    bits=rng.choice([2, 3, 4]))
    if kind == "head_layer":
        return dict(kind=kind, n=_log(rng, 1, 16), h=_log(rng, 16, 110), w=_log(rng, 16, 170),
                    bits=rng.choice([2, 3, 4, 8]))
    if kind == "detector":
        h, w = _log(rng, 128, 800), _log(rng, 128, 1333)
        return dict(kind=kind, n=_log(rng, 1, 8), h=h, w=w, w_pad=(w + 31) // 32 * 32)
    if kind == "eltwise":
        return dict(kind=kind, n=_log(rng, 1, 16), h=_log(rng, 7, 110), w=_log(rng, 7, 180),
                    c=rng.choice([64, 96, 128, 256, 512]), bits=rng.choice([2, 3, 4, 8]),
                    skip_bits=rng.choice([2, 4, 8]))
    if kind == "codes":
        return dict(kind=kind, n=_log(rng, 1, 8), h=_log(rng, 15, 400), w=_log(rng, 15, 672),
                    c=32 * rng.choice([1, 2, 3, 4]), bits=rng.choice([2, 3, 4, 8]))
    if kind == "fake_quant":
        weight = rng.random() < 0.4
        return dict(kind=kind, numel=_log(rng, 4000, 3_000_000 if weight else 60_000_000), bits=rng.randint(2, 8),
                    weight=weight)
    return dict(kind=kind, n=_log(rng, 1, 16), h=_log(rng, 16, 110), w=_log(rng, 16, 170),
                c=rng.choice([64, 96, 256, 320]), levels=rng.randint(1, 5))


def _pyramid(case, levels=5):
    """P3..P7 of a head: every level half the one before, rounded up."""
    h, w = case["h"], case["w"]
    out = []
    for _ in range(levels):
        out.append((h, w))
        h, w = (h + 1) // 2, (w + 1) // 2
    return out


# ------------------------------------------------------------------ inputs, from the seed alone


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _act(g, shape, bits):
    """Activation codes: half-normal at 4 bits (post-ReLU features), uniform otherwise."""
    if bits == 4:
        return (torch.randn(shape, generator=g, device=DEV) * 4).abs_().add_(0.5).floor_().clamp_(0, 15).to(torch.int32)
    return torch.randint(0, 1 << bits, shape, generator=g, device=DEV, dtype=torch.int32)


def _weight(g, shape, bits):
    lim = (1 << (bits - 1)) - 1
    if bits == 4:
        return (torch.randn(shape, generator=g, device=DEV) * 2).add_(0.5).floor_().clamp_(-lim, lim).to(torch.int32)
    return torch.randint(-lim, lim + 1, shape, generator=g, device=DEV, dtype=torch.int32)


def _acc_std(bits, k_total):
    """The accumulator's standard deviation for those draws."""
    if bits == 4:
        return math.sqrt(k_total * 64.0)
    lim, hi = (1 << (bits - 1)) - 1, (1 << bits) - 1
    ex2 = sum(v * v for v in range(hi + 1)) / (hi + 1)
    ew2 = sum(v * v for v in range(-lim, lim + 1)) / (2 * lim + 1)
    return math.sqrt(k_total * ex2 * ew2)


class _Layer:
    """One conv: signed weights, tables (numpy, [levels][cout]) and geometry."""

    def __init__(self, g, rng, cin, cout, k, stride, bits, *, levels=1, out_bits=None, skip=None):
        self.w = _weight(g, (cout, k, k, cin), bits)
        self.bits, self.stride, self.pad = bits, stride, k // 2
        self.out_bits = bits if out_bits is None else out_bits
        std = _acc_std(bits, k * k * cin)
        self.m0, self.shift, self.bias = synth.requant_params(rng, levels, cout, calib_std=std,
                                                              out_bits=min(self.out_bits, 8))
        self.c = self.d = None
        if skip == "codes":
            self.c, self.d = synth.skip_params(rng, levels, cout, self.shift)
        elif skip == "acc":
            self.c, self.d = synth.skip_params_acc(rng, levels, cout)
        if self.out_bits == 32:
            self.m0 = self.shift = None

    def on_device(self):
        W = aqd.ConvWeights(self.w, self.bits)
        rq = aqd.RequantParams.from_numpy(self.m0, self.shift, self.bias)
        sp = None if self.c is None else aqd.SkipParams.from_numpy(self.c, self.d)
        return W, rq, sp


def _inputs(case, seed):
    """(tensors, layers) of a case: int32 codes or float32 values on the GPU, drawn from the seed."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    kind = case["kind"]
    b = case.get("bits")
    if kind == "conv":
        return ([_act(g, (case["n"], case["h"], case["w"], case["cin"]), b)],
                [_Layer(g, rng, case["cin"], case["cout"], case["k"], case["stride"], b)])
    if kind == "bottleneck":
        wide, mid = case["wide"], case["mid"]
        return ([_act(g, (case["n"], case["h"], case["w"], wide), b)],
                [_Layer(g, rng, wide, mid, 1, 1, b), _Layer(g, rng, mid, mid, 3, 1, b),
                 _Layer(g, rng, mid, wide, 1, 1, b, skip="codes")])
    if kind == "down_block":
        ci, co = case["cin"], case["cout"]
        return ([_act(g, (case["n"], case["h"], case["w"], ci), b)],
                [_Layer(g, rng, ci, co, 3, 2, b), _Layer(g, rng, ci, co, 1, 2, b, out_bits=32),
                 _Layer(g, rng, co, co, 3, 1, b, skip="acc")])
    if kind in ("head", "head_layer"):
        lv = _pyramid(case)
        xs = [_act(g, (case["n"], h, w, 256), b) for h, w in lv]
        layers = [_Layer(g, rng, 256, 256, 3, 1, b, levels=len(lv)) for _ in range(case.get("layers", 1))]
        if kind == "head":  # classes and box offsets as one 256 -> 84 conv with int32 outputs
            layers.append(_Layer(g, rng, 256, 84, 3, 1, b, levels=len(lv), out_bits=32))
        return xs, layers
    if kind == "eltwise":
        n, h, w, c, sb = case["n"], case["h"], case["w"], case["c"], case["skip_bits"]
        acc = torch.randint(-20000, 20000, (n, h, w, c), generator=g, device=DEV, dtype=torch.int32)
        same = _act(g, (n, h, w, c), sb)
        coarse = _act(g, (n, (h + 1) // 2, (w + 1) // 2, c), sb)
        t = synth.requant_params(rng, 1, c, calib_std=8000.0, out_bits=b)
        return [acc, same, coarse], [t, synth.skip_params(rng, 1, c, t[1])]
    if kind == "codes":
        return [_act(g, (case["n"], case["h"], case["w"], case["c"]), b)], []
    if kind == "fake_quant":
        n = case["numel"]
        if case["weight"]:
            x, nu = torch.randn(n, generator=g, device=DEV) * 0.6, 0.9
        else:
            x, nu = torch.randn(n, generator=g, device=DEV) * 1.2 + 1.0, 2.5
        gy = torch.randn(n, generator=g, device=DEV) + 0.1
        return [x, gy], [float(np.float32(nu))]
    assert kind == "bn_stats"
    mean = torch.randn(case["c"], generator=g, device=DEV) * 0.5
    return [torch.randn((case["n"], h, w, case["c"]), generator=g, device=DEV) * 2.0 + mean
            for h, w in _pyramid(case, case["levels"])], []


def _network(case, seed):
    return synth.config3(seed, case["n"], case["h"], case["w"], case["w_pad"])


# ------------------------------------------------------------------ the package's calls


def _out(x, layer, W):
    h, w = aqd.conv_out_hw(x.h, x.w, W.kh, W.kw, layer.stride, layer.pad)
    return aqd.DTensor.empty(x.n, h, w, W.cout, layer.out_bits)


def _zeroed(ws):
    return None if ws is None else ws.zero_()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "detector":
        wl = _network(case, seed)
        img = aqd.DTensor.from_codes(torch.from_numpy(wl.inputs[0]).to(DEV), 8)
        return dict(kind=kind, net=IntDetector(wl.extra["layers"], (img.n, img.h, img.w, 3, 8)), img=img)
    ts, layers = _inputs(case, seed)
    st = dict(kind=kind)
    b = case.get("bits")
    if kind == "conv":
        W, rq, _ = layers[0].on_device()
        x = aqd.DTensor.from_codes(ts[0], b)
        y = _out(x, layers[0], W)
        ly = layers[0]
        st.update(x=x, y=y, w=W, rq=rq, stride=ly.stride, pad=ly.pad,
                  ws=aqd.workspace_for([(x, y, None, 0)], W, ly.stride, ly.pad))
    elif kind == "bottleneck":
        p = [ly.on_device() for ly in layers]
        x = aqd.DTensor.from_codes(ts[0], b)
        t1 = _out(x, layers[0], p[0][0])
        t2 = _out(t1, layers[1], p[1][0])
        y = _out(t2, layers[2], p[2][0])
        ws = [_zeroed(aqd.workspace_for([(t, None, None, 0)], p[i][0], 1, layers[i].pad))
              for i, t in enumerate((x, t1, t2))]
        st.update(x=x, t1=t1, t2=t2, y=y, p=p, ws=ws)
    elif kind == "down_block":
        p = [ly.on_device() for ly in layers]
        x = aqd.DTensor.from_codes(ts[0], b)
        a, down = _out(x, layers[0], p[0][0]), _out(x, layers[1], p[1][0])
        y = _out(a, layers[2], p[2][0])
        st.update(x=x, a=a, down=down, y=y, p=p, ws=aqd.workspace_for([(a, y, None, 0)], p[2][0], 1, 1))
    elif kind == "head":
        xs = [aqd.DTensor.from_codes(t, b) for t in ts]
        p = [ly.on_device() for ly in layers]
        jobs, cur = [], xs
        for ly, (W, _, _) in zip(layers, p):
            nxt = [_out(x, ly, W) for x in cur]
            jobs.append([(x, y, None, l) for l, (x, y) in enumerate(zip(cur, nxt))])
            cur = nxt
        ws = aqd.workspace_for(jobs[0], p[0][0], 1, 1)
        sync = torch.zeros(max(4, aqd.tower_sync_bytes(jobs[0], len(jobs), 1)), dtype=torch.uint8, device=DEV)
        st.update(jobs=jobs, ws=[w for w, _, _ in p], rqs=[r for _, r, _ in p], ws_a=ws, ws_b=torch.zeros_like(ws),
                  sync=sync)
    elif kind == "head_layer":
        W, rq, _ = layers[0].on_device()
        jobs = []
        for l, t in enumerate(ts):
            x = aqd.DTensor.from_codes(t, b)
            jobs.append((x, _out(x, layers[0], W), None, l))
        st.update(jobs=jobs, w=W, rq=rq, ws=aqd.workspace_for(jobs, W, 1, 1))
    elif kind == "eltwise":
        (m0, sh, bias), (c, d) = layers
        acc = aqd.DTensor.from_codes(ts[0], 32)
        same, coarse = (aqd.DTensor.from_codes(t, case["skip_bits"]) for t in ts[1:])
        st.update(acc=acc, same=same, coarse=coarse, rq=aqd.RequantParams.from_numpy(m0, sh, bias),
                  sp=aqd.SkipParams.from_numpy(c, d), up=aqd.SkipParams.from_numpy(c, d, upsample=2),
                  y=[aqd.DTensor.empty(acc.n, acc.h, acc.w, acc.c, b) for _ in range(3)])
    elif kind == "codes":
        n, h, w, c = ts[0].shape
        x = aqd.DTensor.empty(n, h, w, c, b)
        ho, wo = aqd.conv_out_hw(h, w, 3, 3, 2, 1)
        st.update(codes=ts[0], x=x, y=aqd.DTensor.empty(n, ho, wo, c, b))
    elif kind == "fake_quant":
        st.update(x=ts[0], gy=ts[1], nu=layers[0], bits=b, weight=case["weight"])
    else:
        st.update(zs=ts)
    return st


def run(state):
    kind = state["kind"]
    if kind == "conv":
        aqd.conv_int(state["x"], state["w"], state["stride"], state["pad"], state["y"], rq=state["rq"],
                     workspace=state["ws"])
        return state["y"].data
    if kind == "bottleneck":
        x, t1, t2, y, ws = state["x"], state["t1"], state["t2"], state["y"], state["ws"]
        (w0, r0, _), (w1, r1, _), (w2, r2, sp) = state["p"]
        aqd.conv_expand_input([(x, None, None, 0)], w0, 1, 0, ws[0])
        aqd.conv_int_grouped_chain([(x, t1, None, 0)], w0, 1, 0, rq=r0, workspace=ws[0], next_pad=1,
                                   next_workspace=ws[1])
        aqd.conv_int_grouped_chain([(t1, t2, None, 0)], w1, 1, 1, rq=r1, workspace=ws[1], next_pad=0,
                                   next_workspace=ws[2])
        aqd.conv_int_grouped_expanded([(t2, y, x, 0)], w2, 1, 0, rq=r2, sp=sp, workspace=ws[2])
        return [t1.data, t2.data, y.data]
    if kind == "down_block":
        x, a, down, y = state["x"], state["a"], state["down"], state["y"]
        (w0, r0, _), (w1, r1, _), (w2, r2, sp) = state["p"]
        aqd.conv_int(x, w0, 2, 1, a, rq=r0)
        aqd.conv_int(x, w1, 2, 0, down, rq=r1)
        aqd.conv_int(a, w2, 1, 1, y, rq=r2, skip=down, sp=sp, workspace=state["ws"])
        return [a.data, down.data, y.data]
    if kind == "head":
        aqd.conv_int_grouped_tower(state["jobs"], state["ws"], state["rqs"], 1, ws_a=state["ws_a"],
                                   ws_b=state["ws_b"], sync=state["sync"])
        return [y.data for jobs in state["jobs"] for _, y, _, _ in jobs]
    if kind == "head_layer":
        aqd.conv_int_grouped(state["jobs"], state["w"], 1, 1, rq=state["rq"], workspace=state["ws"])
        return [y.data for _, y, _, _ in state["jobs"]]
    if kind == "detector":
        net = state["net"]
        net.forward(state["img"])
        return [net.output(f"{head}.{l}") for head in ("cls", "box") for l in range(5)]
    if kind == "eltwise":
        acc, (y0, y1, y2) = state["acc"], state["y"]
        aqd.requant(acc, state["rq"], y0)
        aqd.residual_add_int(acc, state["same"], state["sp"], y1, rq=state["rq"])
        aqd.residual_add_int(acc, state["coarse"], state["up"], y2, rq=state["rq"])
        return [y0.data, y1.data, y2.data]
    if kind == "codes":
        x, y = state["x"], state["y"]
        aqd.pack_codes(state["codes"], x.bits, out=x.data)
        aqd.maxpool_codes(x, 3, 2, 1, y)
        return [x.data, y.data, y.codes()]
    if kind == "fake_quant":
        x, nu, bits, weight = state["x"], state["nu"], state["bits"], state["weight"]
        y, codes = aqd.fake_quant(x, nu, bits, weight=weight)
        gx, gnu = aqd.fake_quant_backward(x, state["gy"], nu, bits, weight=weight)
        return dict(y=y, codes=codes, gx=gx, gnu=gnu)
    return list(aqd.bn_level_stats(state["zs"]))


# ------------------------------------------------------------------ what a pass cannot do without


def _conv_work(n, h, w, cin, cout, k, stride, bits, out_bits, skip_bits=0):
    ho, wo = (h + 2 * (k // 2) - k) // stride + 1, (w + 2 * (k // 2) - k) // stride + 1
    px = n * ho * wo
    return (n * h * w * cin * bits / 8 + cout * k * k * cin * bits / 8 + px * cout * (out_bits + skip_bits) / 8,
            2 * px * cout * k * k * cin)


def _total(parts):
    return {"bytes": int(sum(p[0] for p in parts)), "flops": int(sum(p[1] for p in parts))}


def work(case):
    kind, b = case["kind"], case.get("bits")
    if kind == "conv":
        return _total([_conv_work(case["n"], case["h"], case["w"], case["cin"], case["cout"], case["k"],
                                  case["stride"], b, b)])
    if kind == "bottleneck":
        n, h, w, wide, mid = (case[k] for k in ("n", "h", "w", "wide", "mid"))
        return _total([_conv_work(n, h, w, wide, mid, 1, 1, b, b), _conv_work(n, h, w, mid, mid, 3, 1, b, b),
                       _conv_work(n, h, w, mid, wide, 1, 1, b, b, b)])
    if kind == "down_block":
        n, h, w, ci, co = (case[k] for k in ("n", "h", "w", "cin", "cout"))
        ho, wo = (h + 1) // 2, (w + 1) // 2
        return _total([_conv_work(n, h, w, ci, co, 3, 2, b, b), _conv_work(n, ho, wo, ci, co, 1, 1, b, 32),
                       _conv_work(n, ho, wo, co, co, 3, 1, b, b, 32)])
    if kind in ("head", "head_layer"):
        parts = []
        for h, w in _pyramid(case):
            parts += [_conv_work(case["n"], h, w, 256, 256, 3, 1, b, b)] * case.get("layers", 1)
            if kind == "head":
                parts.append(_conv_work(case["n"], h, w, 256, 84, 3, 1, b, 32))
        return _total(parts)
    if kind == "detector":
        n, size = case["n"], {"image": (case["h"], case["w_pad"], 3, 8)}
        parts = []

        def conv(src, dst, cin, cout, k, s, out=4, skip=0):
            h, w, _, bits = size[src]
            parts.append(_conv_work(n, h, w, cin, cout, k, s, bits, out, skip))
            size[dst] = ((h + s - 1) // s, (w + s - 1) // s, cout, out)
        conv("image", "c", 3, 64, 7, 2)
        h, w = size["c"][:2]
        size["c"] = ((h + 1) // 2, (w + 1) // 2, 64, 4)
        parts.append((n * 32 * (h * w + size["c"][0] * size["c"][1]), 0))  # the stem's max-pool
        cin = 64
        for stage, cout in enumerate((64, 128, 256, 512), start=1):
            for blk in range(2):
                down = stage > 1 and blk == 0
                conv("c", "a", cin, cout, 3, 2 if down else 1)
                if down:
                    conv("c", "d", cin, cout, 1, 2, 32)
                conv("a", "c", cout, cout, 3, 1, 4, 32 if down else 4)
                cin = cout
            size[stage] = size["c"]
        for stage, cin in ((2, 128), (3, 256), (4, 512)):
            conv(stage, f"m{stage}", cin, 256, 1, 1, 4, 0 if stage == 4 else 1)
            conv(f"m{stage}", f"P{stage + 1}", 256, 256, 3, 1)
        conv(4, "P6", 512, 256, 3, 2)
        conv("P6", "P7", 256, 256, 3, 2)
        for l in range(3, 8):
            for _ in range(4):
                conv(f"P{l}", f"P{l}", 256, 256, 3, 1)
            conv(f"P{l}", "out", 256, 84, 3, 1, 32)
        return _total(parts)
    if kind == "eltwise":
        px, c, sb = case["n"] * case["h"] * case["w"], case["c"], case["skip_bits"]
        return {"bytes": int(px * c * (3 * (4 + b / 8) + 1.25 * sb / 8)), "flops": 3 * px * c}
    if kind == "codes":
        n, c = case["n"], case["c"]
        px, po = n * case["h"] * case["w"], n * ((case["h"] + 1) // 2) * ((case["w"] + 1) // 2)
        return {"bytes": int(px * c * (4 + 2 * b / 8) + po * c * (2 * b / 8 + 4)), "flops": 0}
    if kind == "fake_quant":
        return {"bytes": (9 + 12) * case["numel"], "flops": 0}
    px = sum(case["n"] * h * w for h, w in _pyramid(case, case["levels"]))
    return {"bytes": 4 * px * case["c"], "flops": 3 * px * case["c"]}


def tolerance(case):
    if case["kind"] == "fake_quant":
        # A code is decided in float32, so a value at a rounding threshold may take its other
        # neighbour, a whole step away. With the division x / nu replaced by a product with 1 / nu
        # (3e6 to 4e7 values, 2 to 8 bits): y 3e-5, the interval's gradient 3e-5, codes 4e-9 Q.
        return {"rel": 1.2e-4, "differ": 2e-8 * (1 << case["bits"])}
    if case["kind"] == "bn_stats":
        return {"rel": 2e-7}  # float32 runs of 32 values against float64: 3e-8 to 4e-8
    return "exact"


# ------------------------------------------------------------------ the same results in 64 bits


def _table(a):
    return None if a is None else torch.from_numpy(np.asarray(a)).to(DEV).to(torch.int64)


def _rhu(v, r):
    """floor((v + 2^(r-1)) / 2^r), v itself for r = 0."""
    return torch.where(r > 0, (v + (torch.ones_like(r) << (r - 1).clamp(min=0))) >> r, v)


def _finish(t, m0, shift, out_bits):
    u = t.clamp_(-(1 << 31), (1 << 31) - 1)
    if out_bits == 32:
        return u.to(torch.int32)
    return _rhu(u * m0, 31 + shift).clamp_(0, (1 << out_bits) - 1).to(torch.int32)


def _conv64(x, w, stride, pad, level, tables, out_bits, skip=None, upsample=1):
    """Conv of integer codes (NHWC) in float64, the epilogue in int64; int32 codes out."""
    m0, shift, bias, c, d = (None if t is None else _table(t)[level] for t in tables)
    n, h, wd, cin = x.shape
    w = torch.as_tensor(w).to(DEV)
    cout, kh, kw, _ = w.shape
    ho, wo = (h + 2 * pad - kh) // stride + 1, (wd + 2 * pad - kw) // stride + 1
    out = torch.empty((n, ho, wo, cout), dtype=torch.int32, device=DEV)
    w64 = w.to(torch.float64)
    for i in range(n):
        xp = torch.zeros((h + 2 * pad, wd + 2 * pad, cin), dtype=torch.float64, device=DEV)
        xp[pad:pad + h, pad:pad + wd] = x[i]
        acc = torch.zeros((ho * wo, cout), dtype=torch.float64, device=DEV)
        for r in range(kh):
            for s in range(kw):
                tap = xp[r:r + stride * (ho - 1) + 1:stride, s:s + stride * (wo - 1) + 1:stride]
                acc.addmm_(tap.reshape(ho * wo, cin), w64[:, r, s].T)
        t = acc.to(torch.int64).reshape(ho, wo, cout) + bias
        if skip is not None:
            t += _rhu(_up(skip[i:i + 1].to(torch.int64), ho, wo, upsample)[0] * c, d)
        out[i] = _finish(t, m0, shift, out_bits)
    return out


def _up(s, h, w, upsample):
    if upsample == 2:
        s = s.repeat_interleave(2, 1).repeat_interleave(2, 2)
    return s[:, :h, :w]


def _layer64(x, ly, level=0, skip=None):
    return _conv64(x, ly.w, ly.stride, ly.pad, level, (ly.m0, ly.shift, ly.bias, ly.c, ly.d), ly.out_bits, skip)


def _pool64(x, k, stride, pad):
    v = torch.nn.functional.max_pool2d(x.permute(0, 3, 1, 2).to(torch.float64), k, stride, pad)
    return v.permute(0, 2, 3, 1).to(torch.int32).contiguous()


def _packed(codes, bits):
    """int32 codes [..., c] as the bytes of the package's packed rows."""
    if bits == 32:
        return codes.contiguous().view(torch.uint8).reshape(*codes.shape[:-1], -1)
    if bits == 8:
        return codes.to(torch.uint8)
    lead, c = codes.shape[:-1], codes.shape[-1]
    low = bits if bits != 3 else 2
    q = 32 // low

    def words(v, per, width):  # [..., words, per / 4, 4] fields of `width` bits -> bytes
        f = v.reshape(*lead, -1, per // 4, 4)
        sh = torch.arange(per // 4, device=DEV, dtype=torch.int32).mul_(width).reshape(-1, 1)
        return (f << sh).sum(-2).to(torch.uint8)
    if bits != 3:
        return words(codes, q, bits).reshape(*lead, -1)
    lo = words(codes & 3, 16, 2).reshape(*lead, c // 32, 8)
    hi = words(codes >> 2, 32, 1).reshape(*lead, c // 32, 4)
    return torch.cat([lo, hi], -1).reshape(*lead, -1)


def exact(case, seed):
    kind, b = case["kind"], case.get("bits")
    if kind == "detector":
        wl = _network(case, seed)
        t = {"image": torch.from_numpy(wl.inputs[0]).to(DEV)}
        for ly in wl.extra["layers"]:
            if ly.pool is not None:
                t[ly.dst[0]] = _pool64(t[ly.src[0]], *ly.pool)
                continue
            cv = ly.conv
            for l, (s, d) in enumerate(zip(ly.src, ly.dst)):
                t[d] = _conv64(t[s], cv.w, cv.stride, cv.pad, l, (cv.m0, cv.shift, cv.bias, cv.skip_c, cv.skip_d),
                               cv.out_bits, t[ly.skip[l]] if ly.skip else None, ly.upsample)
        return [t[f"{head}.{l}"] for head in ("cls", "box") for l in range(5)]
    ts, layers = _inputs(case, seed)
    if kind == "conv":
        return _packed(_layer64(ts[0], layers[0]), b)
    if kind == "bottleneck":
        t1 = _layer64(ts[0], layers[0])
        t2 = _layer64(t1, layers[1])
        return [_packed(t, b) for t in (t1, t2, _layer64(t2, layers[2], skip=ts[0]))]
    if kind == "down_block":
        a, down = _layer64(ts[0], layers[0]), _layer64(ts[0], layers[1])
        return [_packed(a, b), _packed(down, 32), _packed(_layer64(a, layers[2], skip=down), b)]
    if kind in ("head", "head_layer"):
        out, cur = [], ts
        for ly in layers:
            cur = [_layer64(x, ly, l) for l, x in enumerate(cur)]
            out += [_packed(y, ly.out_bits) for y in cur]
        return out
    if kind == "eltwise":
        (m0, sh, bias), (c, d) = ([_table(t)[0] for t in ts_] for ts_ in layers)
        acc, same, coarse = (t.to(torch.int64) for t in ts)
        h, w = case["h"], case["w"]
        return [_packed(_finish(acc + bias + (0 if s is None else _rhu(_up(s, h, w, u) * c, d)), m0, sh, b), b)
                for s, u in ((None, 1), (same, 1), (coarse, 2))]
    if kind == "codes":
        pooled = _pool64(ts[0], 3, 2, 1)
        return [_packed(ts[0], b), _packed(pooled, b), pooled]
    if kind == "fake_quant":
        x, gy = (t.to(torch.float64) for t in ts)
        nu, q = layers[0], float((1 << b) - 1)
        v = x / nu
        if case["weight"]:
            eta = ((v.clamp(-1, 1) + 1) / 2 * q + 0.5).floor_()
            y, inside, lowest = (2 * eta / q - 1) * nu, (v > -1) & (v < 1), -1.0
            slope = 2 * eta / q - 1 - v
        else:
            eta = (v.clamp(0, 1) * q + 0.5).floor_()
            y, inside, lowest = eta * (nu / q), (v > 0) & (v < 1), 0.0
            slope = eta / q - v
        slope = torch.where(inside, slope, torch.where(v >= 1, 1.0, lowest))
        return dict(y=y, codes=eta.to(torch.uint8), gx=gy * inside, gnu=(gy * slope).sum().reshape(1))
    mean = [z.to(torch.float64).mean((0, 1, 2)) for z in ts]
    var = [((z.to(torch.float64) - m) ** 2).mean((0, 1, 2)) for z, m in zip(ts, mean)]
    return [torch.stack(mean), torch.stack(var)]
