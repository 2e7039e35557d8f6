"""Stages 1 and 2 of the assignment pipeline (Sec. 3.5, pipeline figure): every non-linear layer is run with each
candidate approximation function on calibration activations, scored with the Unified Metric of Eqs. (16)-(20), and
given the candidate with the largest term.

All arithmetic runs in the library: one ``iptq_analyze_*`` launch per layer evaluates the float layer and every integer
candidate (on the device functions of the deployed kernels) and reduces their error sums, the scoring is
``iptq_metric_term`` / ``iptq_metric_select``.  This module only sequences the calls and keeps the results; it
synchronises with the device once, in ``finish()``.
"""
from __future__ import annotations

from dataclasses import dataclass, field

import numpy as np
import torch

from . import api

SOFTMAX_CANDIDATES = (api.SM_BITEXP, api.SM_SHIFTMAX, api.SM_POLY, api.SM_LOG2)
GELU_CANDIDATES = (api.GELU_POLY4, api.GELU_POLY2, api.GELU_SHIFT)
LN_CANDIDATES = (api.LN_SHIFT, api.LN_NEWTON, api.LN_PTF)


@dataclass
class Candidate:
    variant: int
    op_count: float
    slot: int                      # row of the device sums buffer
    sum_x2: float = float("nan")
    sum_err2: float = float("nan")
    sqnr_db: float = float("nan")
    perturbation: float = float("nan")
    term: float = float("nan")


@dataclass
class Layer:
    name: str
    kind: int
    candidates: list = field(default_factory=list)
    choice: int = -1               # variant id of the selected candidate


class Analyzer:
    def __init__(self, device="cuda", max_evaluations=256, c_unit=1.0e6):
        self.device = device
        self.c_unit = float(c_unit)
        self.max_evaluations = max_evaluations
        # the scratch of the launches (its counter starts at zero) and the sums, with room for one more layer's candidates
        # behind the last evaluation that counts
        self._buf = torch.empty(api.ANALYZE_WORK_BYTES // 8 + 2 * (max_evaluations + api.ANALYZE_MAX_CANDIDATES), dtype=torch.float64,
                                device=device)
        self._buf[0] = 0
        self.sums = self._buf[api.ANALYZE_WORK_BYTES // 8:].view(-1, 2)
        self._work_ptr, self._sums_ptr = self._buf.data_ptr(), self.sums.data_ptr()
        self._native = api.native()
        self.layers: list[Layer] = []
        self.n_eval = 0

    def _add(self, layer, variants, launch, per_launch=api.ANALYZE_MAX_CANDIDATES):
        """Runs the candidates of one layer, as many per launch as a launch takes, and records them."""
        variants = tuple(variants)
        for i in range(0, len(variants), per_launch):
            # a launch that goes past the capacity writes its sums into the room behind it
            done = launch(variants[i:i + per_launch], self._sums_ptr + 16 * self.n_eval, self._work_ptr)
            for v, ops in done:
                if self.n_eval >= self.max_evaluations:
                    raise RuntimeError("more evaluations than max_evaluations")
                layer.candidates.append(Candidate(v, ops, self.n_eval))
                self.n_eval += 1
        self.layers.append(layer)
        return layer

    def softmax_layer(self, name, scores, in_scale, variants=SOFTMAX_CANDIDATES, out_bits=8):
        """scores: device int32 [rows, n] at scale in_scale.  A candidate that has no integer constants at this scale is left
        out."""
        n = self._native
        return self._add(Layer(name, api.LAYER_SOFTMAX), variants,
                         lambda v, sums, work: n.analyze_softmax(scores, in_scale, v, out_bits, sums, work))

    def gelu_layer(self, name, x, in_scale, in_bits, out_scale, out_zp, variants=GELU_CANDIDATES, out_bits=8):
        """x: device int32 (any shape) at scale in_scale, in_bits wide.  A candidate that has no integer constants at this scale
        and width is left out."""
        n = self._native
        return self._add(Layer(name, api.LAYER_GELU), variants,
                         lambda v, sums, work: n.analyze_gelu(x, in_scale, in_bits, out_scale, out_zp, out_bits, v, sums, work), 3)

    def layernorm_layer(self, name, x, gamma, beta, out_scale, out_zp, variants=LN_CANDIDATES, ptf_shift=None,
                        out_bits=8):
        """x: device int8 [rows, dim]; gamma, beta: host float32 [dim]; ptf_shift: device uint8 [dim], used by the
        LN_PTF candidate only (the other candidates read x as it is; without it the LN_PTF candidate is left out)."""
        n = self._native
        g, b = np.ascontiguousarray(gamma, dtype=np.float32), np.ascontiguousarray(beta, dtype=np.float32)
        return self._add(Layer(name, api.LAYER_LAYERNORM), variants,
                         lambda v, sums, work: n.analyze_layernorm(x, g, b, out_scale, out_zp, out_bits, v, ptf_shift, sums, work))

    def finish(self):
        """Reads the sums back (the only synchronisation), scores every candidate and selects per layer.
        Returns (layers, Omega) with Omega the sum of the selected terms, Eq. (16)."""
        host = self.sums[:max(self.n_eval, 1)].cpu()
        ptr = host.data_ptr()
        omega = 0.0
        for layer in self.layers:
            cands = layer.candidates
            best, scores = self._native.metric_scores(ptr, cands[0].slot if cands else 0, [c.op_count for c in cands], self.c_unit)
            for cand, (cand.sum_x2, cand.sum_err2, cand.sqnr_db, cand.term) in zip(cands, scores):
                cand.perturbation = cand.sum_err2
            layer.choice = cands[best].variant
            omega += cands[best].term
        return self.layers, omega


def block_tables(layers, n_blocks):
    """Per-block (softmax, gelu, ln1, ln2) variant tuples from layers named 'blk{i}.{ln1|softmax|ln2|gelu}'."""
    by_name = {l.name: l.choice for l in layers}
    return [(by_name["blk%d.softmax" % i], by_name["blk%d.gelu" % i], by_name["blk%d.ln1" % i],
             by_name["blk%d.ln2" % i]) for i in range(n_blocks)]
