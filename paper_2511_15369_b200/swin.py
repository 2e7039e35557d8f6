"""Swin-shaped backbone as a sequence of C-ABI calls: per block the integer encoder block with the window index of its
7x7 windows (cyclic shift and padding folded into the table; relative-position bias, attention labels), so that tokens stay in
grid order between blocks; between stages the 2x2 patch merge (integer LayerNorm of gathered rows, INT8 linear).
Host logic only: tables and parameters are prepared once, every step of the data path runs in the library."""
from __future__ import annotations

import numpy as np
import torch

from . import api


class SwinBackbone:
    def __init__(self, spec, table=(api.SM_BITEXP, api.GELU_POLY4, api.LN_SHIFT, api.LN_SHIFT), device="cuda"):
        self.spec = spec
        self.layers = []
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(device)
        for st in spec.stages:
            C = st["dim"]
            for bspec, shift, fwd, rev in st["blocks"]:
                self.layers.append(("block", api.EncoderBlock(bspec, table, device, window_index=dev(fwd.reshape(-1)),
                                                              grid_rows=rev.size)))
            if st["merge"] is not None:
                m, tab = st["merge"]
                gq, bq, lc = api.layernorm_prepare(m.gamma, m.beta, m.ln_out_scale, 0)
                mult, shift = api.channel_requant_prepare(m.ratio)
                ws = api.Workspace(api.linear_workspace_bytes(tab.shape[0], 2 * C, 4 * C))
                self.layers.append(("merge", dev(tab), dev(gq), dev(bq), lc, dev(m.w), dev(mult), dev(shift), ws))

    def __call__(self, x):
        for L in self.layers:
            if L[0] == "block":
                x = L[1](x)
            else:
                _, tab, gq, bq, lc, w, mult, shift, ws = L
                h = api.layernorm_gather(x, tab, gq, bq, lc)
                x = api.linear(h, w, None, mult, shift, ws)
        return x

    def check(self):
        for L in self.layers:
            (L[1].ws if L[0] == "block" else L[8]).check()

    def gemm_ops(self) -> int:
        ops = 0
        for st in self.spec.stages:
            for bspec, _, _, rev in st["blocks"]:
                # LN1, QKV and the attention run on window rows, padding included; the layers behind them on the grid's tokens
                s = bspec.shape
                ops += s.gemm_ops() - 2 * (s.T - rev.size) * (s.D * s.D + 2 * s.D * s.Dh)
            if st["merge"] is not None:
                m, tab = st["merge"]
                ops += 2 * tab.shape[0] * m.w.shape[0] * m.w.shape[1]
        return ops
