"""The calls this library is used for, as timed cases: the stand-alone integer non-linears, the fused encoder block,
the whole models composed of it and the Unified-Metric analysis.

Every case is one pass through the public Python entry points (``paper_2511_15369_b200.api`` / ``vit`` / ``swin`` /
``assign``), called the plain way: eagerly, on the current stream.  The path is inference only, so there is one
direction.  Sizes are those of ``synth.CONFIGS``, ``synth.SWIN_T_STAGES`` and ``synth.VIT_MODELS``, the distributions
those of ``synth`` drawn on the device (logits N(0, 3^2) with 1 % of a row at +12, GELU inputs N(-0.3, 1.2^2) with a
0.5 % Laplace tail, LayerNorm inputs N(0, 1) with 2 % of the channels x20, weights N(0, 0.02^2)).  Weights and scales
are calibrated on the host by ``synth`` on a few images; a model's blocks share two sets of values (each block has
its own device copy, so the traffic is that of different weights).
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2511_15369_b200 import api, assign, swin, synth, vit

SM = {"bitexp": api.SM_BITEXP, "shiftmax": api.SM_SHIFTMAX, "poly": api.SM_POLY, "log2": api.SM_LOG2}
GELU = {"poly4": api.GELU_POLY4, "poly2": api.GELU_POLY2, "shift": api.GELU_SHIFT}
LN = {"shift": api.LN_SHIFT, "newton": api.LN_NEWTON, "ptf": api.LN_PTF}
SCALES = {"acc": synth.SOFTMAX_SCALE_ACC, "8bit": synth.SOFTMAX_SCALE_8BIT}


def listed():
    block = dict(kind="block", w_bits=8, sm="bitexp", gelu="poly4", ln1="shift", ln2="shift", grid=0, shift=0)
    return [
        # The smallest calls: the three non-linears of one DeiT-Tiny block for a single image, one call each.
        dict(name="nonlinears_tiny_b1", kind="nonlinears", B=1, N=197, D=192, H=3, sm="bitexp", gelu="poly4", ln="shift"),
        # The stand-alone non-linears on tensors of batch inference, larger than the L2 cache.
        dict(name="softmax_base_b128", kind="softmax", rows=128 * 12 * 197, n=197, sm="bitexp", scale="acc", period=0),
        dict(name="gelu_base_b128", kind="gelu", elems=128 * 197 * 3072, gelu="poly4", in_bits=16, table=True),
        dict(name="layernorm_base_b1024", kind="layernorm", rows=1024 * 197, dim=768, ln="shift"),
        # Choosing the approximation of every layer from calibration activations: 12 blocks of DeiT-Small, 8 images.
        dict(name="analysis_small_b8", kind="analysis", B=8, N=197, D=384, H=6, depth=12),
        # One encoder block: a single image (latency), medium and large batches, 4-bit weights unpacked in the call,
        # shifted windows with relative-position bias and labels.
        dict(block, name="block_tiny_b1", B=1, N=197, D=192, H=3),
        dict(block, name="block_small_b64", B=64, N=197, D=384, H=6),
        dict(block, name="block_base_b128", B=128, N=197, D=768, H=12),
        dict(block, name="block_base_w4_b8", B=8, N=197, D=768, H=12, w_bits=4, sm="shiftmax", gelu="poly2"),
        dict(block, name="block_swin_b64", B=64, N=49, D=96, H=3, grid=56, shift=3),
        # Whole models: the latency table's batch of 8, and the detection backbone (two images, 200 x 304 tokens).
        dict(name="vit_small_b8", kind="vit", model="DeiT-S", B=8, img=224),
        dict(name="swin_tiny_800x1216_b2", kind="swin", B=2, h=200, w=304),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["nonlinears", "softmax", "gelu", "layernorm", "analysis", "block", "block", "block", "windows",
                       "vit", "swin"])
    sm, gelu = rng.choice(list(SM)), rng.choice(list(GELU))
    ln = [rng.choice(list(LN)) for _ in range(2)]
    if kind == "nonlinears":
        H = rng.choice([3, 6, 12])
        return dict(kind=kind, B=rng.randint(1, 8), N=rng.randint(17, 256), D=64 * H, H=H, sm=sm, gelu=gelu, ln=ln[0])
    if kind == "softmax":
        # attention scores: windows (bias rows repeat per window, each head its own) to long sequences
        n = rng.choice([49, 64, 197, 257, int(_log(rng, 16, 1024))])
        rows = max(1, int(_log(rng, 1e5, 5.9e7) / n))
        return dict(kind=kind, rows=rows, n=n, sm=sm, scale=rng.choice(list(SCALES)), period=rng.choice([0, 0, 3 * n]))
    if kind == "gelu":
        return dict(kind=kind, elems=int(_log(rng, 1e5, 7.7e7)), gelu=gelu, in_bits=rng.choice([8, 12, 16]),
                    table=rng.random() < 0.5)
    if kind == "layernorm":
        dim = rng.choice([96, 192, 384, 768, 1024, 1536, 4 * rng.randint(12, 768)])
        return dict(kind=kind, rows=max(1, int(_log(rng, 1e5, 1.5e8) / dim)), dim=dim, ln=ln[0])
    if kind == "analysis":
        H = rng.choice([3, 6])
        return dict(kind=kind, B=rng.randint(1, 8), N=rng.choice([50, 145, 197]), D=64 * H, H=H, depth=rng.randint(1, 12))
    if kind == "block":
        H = rng.choice([3, 6, 12])
        N = rng.choice([50, 101, 145, 197, 197, rng.randint(17, 256)])
        most = 24000 * 768 / (N * 64 * H) if H < 12 else 24000 / N
        return dict(kind="block", B=max(1, int(_log(rng, 1, most))), N=N, D=64 * H, H=H, w_bits=rng.choice([8, 8, 6, 4]),
                    sm=sm, gelu=gelu, ln1=ln[0], ln2=ln[1], grid=0, shift=0)
    if kind == "windows":
        H = rng.choice([3, 6, 12, 24])
        grid = rng.choice([7, 14, 28, 56, rng.randint(8, 60)])
        windows = (-(-grid // 7)) ** 2
        most = max(1.0, 180000 * 96 / (49 * windows * 32 * H))
        return dict(kind="block", B=max(1, int(_log(rng, 1, most))), N=49, D=32 * H, H=H, w_bits=rng.choice([8, 8, 6, 4]),
                    sm=sm, gelu=gelu, ln1=ln[0], ln2=ln[1], grid=grid, shift=rng.choice([0, 3]))
    if kind == "vit":
        return dict(kind=kind, model=rng.choice(list(synth.VIT_MODELS)), B=rng.randint(1, 16), img=rng.choice([160, 192, 224]))
    return dict(kind=kind, B=rng.randint(1, 2), h=rng.randint(40, 200), w=rng.randint(40, 300))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _logits(g, rows, n, scale):
    x = torch.empty((rows, n), device="cuda").normal_(0.0, 3.0, generator=g)
    k = max(1, math.ceil(0.01 * n))
    at = torch.randint(0, n, (rows, k), device="cuda", generator=g)
    return x.scatter_(1, at, 12.0).div_(scale).round_().to(torch.int32)


def _gelu_in(g, n, bits):
    """int32 [n] and the scale of its symmetric quantiser."""
    x = torch.empty(n, device="cuda").normal_(-0.3, 1.2, generator=g)
    tail = torch.rand(n, device="cuda", generator=g) < 0.005
    u = torch.rand(n, device="cuda", generator=g) - 0.5
    x = torch.where(tail, -4.0 * u.sign() * torch.log1p(-2.0 * u.abs().clamp(max=0.499999)), x)
    scale = float(x.abs().max()) / ((1 << (bits - 1)) - 1)
    return x.div_(scale).round_().to(torch.int32), scale


def _ln_in(g, rows, dim, bits=8):
    """int8 [rows, dim] whose large channels are the same for all rows."""
    big = torch.ones(dim, device="cuda")
    big[torch.randperm(dim, device="cuda", generator=g)[:max(1, round(0.02 * dim))]] = 20.0
    x = torch.empty((rows, dim), device="cuda").normal_(0.0, 1.0, generator=g).mul_(big)
    q = (1 << (bits - 1)) - 1
    return x.mul_(q / float(x.abs().max())).round_().to(torch.int8)


def _ln_params(seed, dim):
    r = np.random.default_rng(seed)
    return r.normal(1.0, 0.1, dim).astype(np.float32), r.normal(0.0, 0.1, dim).astype(np.float32)


def _ptf(x):
    return torch.from_numpy(synth.ptf_shifts(x[:256].cpu().numpy())).cuda()


LN_OUT_SCALE = 8.0 / 127.0          # eight standard deviations
GELU_OUT = (8.2 / 255.0, -123)      # [-0.17, 8]: scale and zero point


def _softmax_consts(scale, n, sm):
    c = api.softmax_prepare(scale, n, 4 if SM[sm] == api.SM_LOG2 else 8, SM[sm])
    return c, api.softmax_table(c)


def _layernorm_state(x, seed, ln):
    gamma, beta = _ln_params(seed, x.shape[1])
    gq, bq, c = api.layernorm_prepare(gamma, beta, LN_OUT_SCALE, 0, 8, LN[ln])
    return dict(x=x, g=torch.from_numpy(gq).cuda(), b=torch.from_numpy(bq).cuda(), c=c,
                ptf=_ptf(x) if LN[ln] == api.LN_PTF else None)


def _gelu_state(g, n, gelu, in_bits, table):
    x, scale = _gelu_in(g, n, in_bits)
    c = api.gelu_prepare(scale, in_bits, GELU_OUT[0], GELU_OUT[1], 8, GELU[gelu])
    return dict(x=x, c=c, keep=api.gelu_table(c) if table else None)


def _block_spec(shape, calib, seed, w_bits=8):
    """A calibrated block of `shape`: weights and scales come from `calib` attention problems."""
    small = synth.make_block(dataclasses.replace(shape, B=calib), seed=seed, w_bits=w_bits, calib_images=calib,
                             a_bits=6 if w_bits == 6 else 8)
    small.shape, small.x = shape, None
    return small


def _prepare_block(case, seed):
    B, mask = case["B"], None
    if case["grid"]:
        _, mask, _, windows = synth.swin_window_tables(B, case["grid"], case["grid"], case["shift"])
        B *= windows
    shape = synth.BlockShape("block", B, case["N"], case["D"], case["H"], case["D"] // case["H"], 4 * case["D"], bool(case["grid"]))
    spec = _block_spec(shape, 2 if case["N"] > 64 else 4, seed, case["w_bits"])
    spec.mask_id = mask if case["shift"] else None
    blk = api.EncoderBlock(spec, (SM[case["sm"]], GELU[case["gelu"]], LN[case["ln1"]], LN[case["ln2"]]))
    return dict(block=blk, x=_ln_in(_gen(seed), shape.T, shape.D, spec.a_bits))


def _prepare_vit(case, seed):
    spec = synth.make_vit(case["model"], case["B"], seed, case["img"], depth=2)
    spec.blocks = spec.blocks * (synth.VIT_MODELS[case["model"]]["depth"] // 2)
    return dict(model=vit.VitModel(spec), image=torch.from_numpy(spec.image).cuda())


def _stages(case):
    h, w = case["h"], case["w"]
    for st in synth.SWIN_T_STAGES:
        yield st["dim"], st["heads"], st["depth"], h, w
        h, w = -(-h // 2), -(-w // 2)


def _prepare_swin(case, seed):
    B, stages = case["B"], []
    for i, (C, H, depth, h, w) in enumerate(_stages(case)):
        blocks = []
        for shift in (0, 3):
            fwd, mask, rev, windows = synth.swin_window_tables(B, h, w, shift)
            shape = synth.BlockShape("stage %d" % i, B * windows, 49, C, H, C // H, 4 * C, True)
            spec = _block_spec(shape, 4, seed + 10 * i + shift)
            spec.mask_id = mask
            blocks.append((spec, shift, fwd, rev))
        merge = (synth.make_merge(C, seed + 10 * i + 5), synth.swin_merge_table(B, h, w)) if i < 3 else None
        stages.append(dict(dim=C, heads=H, grid=(h, w), blocks=blocks * (depth // 2), merge=merge))
    return dict(model=swin.SwinBackbone(synth.SwinSpec(B, stages, None)),
                image=_ln_in(_gen(seed), B * case["h"] * case["w"], synth.SWIN_T_STAGES[0]["dim"]))


def _prepare_analysis(case, seed):
    g, B, N, D, H = _gen(seed), case["B"], case["N"], case["D"], case["H"]
    layers = []

    def ln(name, k):
        x = _ln_in(g, B * N, D)
        layers.append(("layernorm", name, x, _ln_params(seed + k, D), _ptf(x)))
    for i in range(case["depth"]):
        ln("blk%d.ln1" % i, 2 * i)
        layers.append(("softmax", "blk%d.softmax" % i, _logits(g, B * H * N, N, synth.SOFTMAX_SCALE_ACC)))
        ln("blk%d.ln2" % i, 2 * i + 1)
        layers.append(("gelu", "blk%d.gelu" % i) + _gelu_in(g, B * N * 4 * D, 16))
    ln("final.ln", 2 * case["depth"])
    return dict(layers=layers)


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    state = dict(case=case)
    if kind == "nonlinears":
        B, N, D, H = case["B"], case["N"], case["D"], case["H"]
        c, keep = _softmax_consts(synth.SOFTMAX_SCALE_ACC, N, case["sm"])
        state.update(softmax=dict(x=_logits(g, B * H * N, N, synth.SOFTMAX_SCALE_ACC), c=c, keep=keep),
                     gelu=_gelu_state(g, B * N * 4 * D, case["gelu"], 16, True),
                     layernorm=_layernorm_state(_ln_in(g, B * N, D), seed, case["ln"]))
    elif kind == "softmax":
        scale = SCALES[case["scale"]]
        c, keep = _softmax_consts(scale, case["n"], case["sm"])
        bias = None
        if case["period"]:
            bias = torch.empty((case["period"], case["n"]), device="cuda").normal_(0.0, 1.0, generator=g).div_(scale).round_().to(torch.int32)
        state.update(x=_logits(g, case["rows"], case["n"], scale), c=c, keep=keep, bias=bias)
    elif kind == "gelu":
        state.update(_gelu_state(g, case["elems"], case["gelu"], case["in_bits"], case["table"]))
    elif kind == "layernorm":
        state.update(_layernorm_state(_ln_in(g, case["rows"], case["dim"]), seed, case["ln"]))
    else:
        state.update({"analysis": _prepare_analysis, "block": _prepare_block, "vit": _prepare_vit, "swin": _prepare_swin}[kind](case, seed))
    return state


# ------------------------------------------------------------------ one pass

def _run_analysis(state):
    an = assign.Analyzer()
    for kind, name, x, *rest in state["layers"]:
        if kind == "softmax":
            an.softmax_layer(name, x, synth.SOFTMAX_SCALE_ACC)
        elif kind == "gelu":
            an.gelu_layer(name, x, rest[0], 16, *GELU_OUT)
        else:
            (gamma, beta), ptf = rest
            an.layernorm_layer(name, x, gamma, beta, LN_OUT_SCALE, 0, ptf_shift=ptf)
    layers, omega = an.finish()
    cands = [c for layer in layers for c in layer.candidates]
    return dict(choices=np.array([layer.choice for layer in layers]), omega=omega, terms=np.array([c.term for c in cands]),
                sum_x2=np.array([c.sum_x2 for c in cands]), sum_err2=np.array([c.sum_err2 for c in cands]))


def run(state):
    kind = state["case"]["kind"]
    if kind == "nonlinears":
        s, e, l = state["softmax"], state["gelu"], state["layernorm"]
        return [api.softmax(s["x"], s["c"]), api.gelu(e["x"], e["c"]), api.layernorm(l["x"], l["g"], l["b"], l["c"], l["ptf"])]
    if kind == "softmax":
        return api.softmax(state["x"], state["c"], state["bias"])
    if kind == "gelu":
        return api.gelu(state["x"], state["c"])
    if kind == "layernorm":
        return api.layernorm(state["x"], state["g"], state["b"], state["c"], state["ptf"])
    if kind == "block":
        return state["block"](state["x"])
    if kind == "analysis":
        return _run_analysis(state)
    return state["model"](state["image"])


# ------------------------------------------------------------------ what a pass cannot do without

def _block_work(T, problems, N, D, w_bits=8):
    """(weight bytes, contraction operations) of an encoder block on T tokens in `problems` attention problems."""
    return 12 * D * D * (4 if w_bits == 4 else 8) / 8, 2 * (12 * T * D * D + 2 * problems * N * N * D)


def work(case):
    """Tensors and weights read and written once; operations are those of the contractions on real tokens (the
    element-wise arithmetic of the non-linears is not counted)."""
    kind = case["kind"]
    if kind == "nonlinears":
        T = case["B"] * case["N"]
        return dict(bytes=5 * T * case["H"] * case["N"] + 5 * 4 * T * case["D"] + 2 * T * case["D"], flops=0)
    if kind == "softmax":
        return dict(bytes=5 * case["rows"] * case["n"] + 4 * case["period"] * case["n"], flops=0)
    if kind == "gelu":
        return dict(bytes=5 * case["elems"], flops=0)
    if kind == "layernorm":
        return dict(bytes=2 * case["rows"] * case["dim"], flops=0)
    if kind == "analysis":
        # every layer's activations once
        T = case["B"] * case["N"]
        per_block = 4 * T * case["H"] * case["N"] + 4 * 4 * T * case["D"] + 2 * T * case["D"]
        return dict(bytes=case["depth"] * per_block + T * case["D"], flops=0)
    if kind == "block":
        problems = case["B"] * (-(-case["grid"] // 7)) ** 2 if case["grid"] else case["B"]
        T = problems * case["N"]
        w, ops = _block_work(T, problems, case["N"], case["D"], case["w_bits"])
        return dict(bytes=w + 2 * T * case["D"], flops=ops)
    if kind == "vit":
        D, depth, B = synth.VIT_MODELS[case["model"]]["D"], synth.VIT_MODELS[case["model"]]["depth"], case["B"]
        P = (case["img"] // 16) ** 2
        w, ops = _block_work(B * (P + 1), B, P + 1, D)
        return dict(bytes=depth * w + 768 * D + 1000 * D + B * (3 * case["img"] ** 2 + 1000),
                    flops=depth * ops + 2 * B * (P * 768 * D + 1000 * D))
    n_bytes, n_ops, B = 0, 0, case["B"]
    for i, (C, H, depth, h, w) in enumerate(_stages(case)):
        wb, ops = _block_work(B * h * w, B * h * w / 49, 49, C)
        n_bytes += depth * wb
        n_ops += depth * ops
        if i == 0:
            n_bytes += B * h * w * C
        if i < 3:
            n_bytes += 8 * C * C
            n_ops += 2 * B * -(-h // 2) * -(-w // 2) * 8 * C * C
        else:
            n_bytes += B * h * w * C
    return dict(bytes=n_bytes, flops=n_ops)


def tolerance(case):
    """Everything is integer and exact, except the fp64 sums of the analysis: another order of summation and another
    fp64 exp / erf move them by a few 1e-13."""
    return {"rel": 1e-9, "max": 1e-8} if case["kind"] == "analysis" else "exact"
