"""The user query's own forward pass and the first decode step over the context cache: what surrounds the repair
loop in the paper's time-to-first-token region (Section 2: the scores come from a pass of the query over the naive
cache, one attention per layer; reproducibility appendix: query prefill and the first token's decode close the timed
region).  Call sequencing over torch buffers only; every operation runs in the CUDA kernels behind
`binding`.

Per layer the query's rows run the decoder block: RMSNorm, the stacked Q/K/V projection, per-head Q/K norm where the
model has one, rotary embedding at positions T_c, T_c + 1, ... and the append of their K/V to the cache behind the context rows (one launch),
then causal attention over [context, query] (`relaxkv_query_prefill_attention`, which can emit the context scores of
that very pass), output projection + residual, MLP + residual.  The decode step is the same block for one new token
(the projections take the streaming one-row kernel), followed by the final norm and the output head.
"""
from __future__ import annotations

from typing import Dict, List, Optional, Sequence

import torch

from . import binding as B
from .inputs import BlockShape


# Layers whose context scores are computed by one launch behind the last of them, and the query rows kept for that (10 MB of Q at 40
# heads of 128).  By itself a layer of few rows is mostly its launch's start and end: 57 rows over 8K of context 15 + 4 us of which 4 are
# work; 8 layers of such a pass took 1321 us, 1278 so, 12 layers of 128 rows over 32K 4264 / 4221.  With more rows a launch is full by itself.
_SCORE_LAYERS, _SCORE_ROWS = 8, 1024


class QueryPass:
    """Buffers for the block work of the query rows of a batch (`q_lens` tokens per request after `ctx_lens` context
    tokens).  The caches handed to `prefill` / `decode` must have room for ctx + query (+ decoded) tokens per request."""

    def __init__(self, n_q_heads: int, n_kv_heads: int, head_dim: int, ctx_lens: Sequence[int], q_lens: Sequence[int],
                 blk: BlockShape, device="cuda", softmax_scale: Optional[float] = None, extra_tokens: int = 1):
        self.blk = blk
        self.ctx_lens, self.q_lens = [int(x) for x in ctx_lens], [int(x) for x in q_lens]
        self.device = torch.device(device)
        H, Hkv, D, C, I = n_q_heads, n_kv_heads, head_dim, blk.hidden, blk.inter
        self.H, self.Hkv, self.D = H, Hkv, D
        nb = len(self.ctx_lens)
        n = sum(self.q_lens)
        bf = dict(dtype=torch.bfloat16, device=self.device)
        i32 = dict(dtype=torch.int32, device=self.device)
        # shapes: context + query (prefill), and + the decoded tokens so far (decode)
        self.shape_prefill = B.Shape(H, Hkv, D, self.ctx_lens, self.q_lens, softmax_scale)
        ext = [c + q for c, q in zip(self.ctx_lens, self.q_lens)]
        self.shape_ext = B.Shape(H, Hkv, D, ext, self.q_lens, softmax_scale)
        self.shape_dec = B.Shape(H, Hkv, D, [e + extra_tokens for e in ext], [1] * nb, softmax_scale)
        nbytes = max(B.relaxkv_workspace_bytes(self.shape_ext, 1), B.relaxkv_workspace_bytes(self.shape_dec, 1))
        ws = torch.empty(nbytes + 256, dtype=torch.uint8, device=self.device)
        off = (-ws.data_ptr()) % 256
        self.workspace = ws[off:off + nbytes]
        e = lambda *s: torch.empty(*s, **bf)
        self.x, self.a, self.h = e(n, C), e(n, C), [e(n, C), e(n, C)]
        self.q, self.k, self.v, self.o = e(n, H, D), e(n, Hkv, D), e(n, Hkv, D), e(n, H, D)
        self.gu, self.m = e(n, 2 * I), e(n, I)
        self.lse = torch.empty(H, n, dtype=torch.float32, device=self.device)
        # rotated queries and row normalisers of the layers that are scored together, as far as the workspace reaches
        g = max(1, min(_SCORE_LAYERS, _SCORE_ROWS // max(1, n)))
        while g > 1 and B.relaxkv_workspace_bytes(self.shape_prefill, g) > nbytes:
            g -= 1
        self.q_kept = torch.empty(g, n, H, D, **bf) if g > 1 else None
        self.lse_kept = torch.empty(g, H, n, dtype=torch.float32, device=self.device) if g > 1 else None
        # positions of the query tokens (request-local) and their offsets: plain index data, built once
        pos, cu = [], [0]
        for c, q in zip(self.ctx_lens, self.q_lens):
            pos.append(torch.arange(c, c + q, dtype=torch.int32))
            cu.append(cu[-1] + q)
        self.q_pos = torch.cat(pos).to(self.device)
        self.q_cu = torch.tensor(cu, **i32)
        self.last_rows = torch.tensor([c - 1 for c in cu[1:]], dtype=torch.long, device=self.device)
        # decode buffers: one row per request
        self.dx, self.da, self.dh = e(nb, C), e(nb, C), [e(nb, C), e(nb, C)]
        self.dq, self.dk, self.dv, self.do = e(nb, H, D), e(nb, Hkv, D), e(nb, Hkv, D), e(nb, H, D)
        self.dgu, self.dm = e(nb, 2 * I), e(nb, I)
        self.d_cu = torch.arange(nb + 1, **i32)
        self._dec_pos = {}

    def decode_positions(self, step: int) -> torch.Tensor:
        """Device tensor of the decoded token's position per request (T_c + Q_b + step), built once per step index so
        that `decode` itself performs no host-to-device copy (it can then be captured into a CUDA graph)."""
        if step not in self._dec_pos:
            self._dec_pos[step] = torch.tensor([c + q + step for c, q in zip(self.ctx_lens, self.q_lens)],
                                               dtype=torch.int32, device=self.device)
        return self._dec_pos[step]

    def _block(self, l, w, cache, h, x, a, q, k, v, o, gu, m, h_out, pos, cu, counts, shape, attend, rec):
        blk, D, n = self.blk, self.D, h.shape[0]
        rec("norm", lambda: B.relaxkv_rmsnorm(h, w["w_in_norm"], x, blk.eps))
        if "w_qkv" not in w:                            # weight-loading step, once per layer: [Wq; Wk; Wv] stacked
            w["w_qkv"] = B.stack_qkv(w["wq"], w["wk"], w["wv"])
        rec("qkv_proj", lambda: B.relaxkv_linear_qkv(x, w["w_qkv"], q, k, v))
        rec("rope_append", lambda: B.relaxkv_qk_norm_rope_append(shape, cache, q, k, v, pos, cu, counts, blk.rope_theta,
                                                                 w.get("w_q_norm"), w.get("w_k_norm"), blk.eps))
        rec("attention", attend)
        rec("o_proj", lambda: B.relaxkv_linear(o, w["wo"], a, residual=h))
        rec("norm", lambda: B.relaxkv_rmsnorm(a, w["w_post_norm"], x, blk.eps))
        if blk.inter % 128 == 0:
            if "w_gate_up_tiled" not in w:              # weight-loading step, once per layer
                w["w_gate_up_tiled"] = B.tile_gate_up(w["w_gate_up"])
            rec("mlp", lambda: B.relaxkv_linear_swiglu(x, w["w_gate_up_tiled"], m))
        else:
            rec("mlp", lambda: (B.relaxkv_linear(x, w["w_gate_up"], gu), B.relaxkv_swiglu(gu, m)))
        rec("mlp", lambda: B.relaxkv_linear(m, w["w_down"], h_out, residual=a))

    @staticmethod
    def _rec(events):
        def rec(name, fn):
            if events is None:
                fn(); return
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(); fn(); b.record(); events.append((name, a, b))
        return rec

    def prefill(self, h0: torch.Tensor, weights: List[Dict[str, torch.Tensor]], caches: List[B.CacheView],
                scores_out: Optional[torch.Tensor] = None, events: Optional[list] = None,
                taps: Optional[list] = None) -> torch.Tensor:
        """h0: input representations of the query tokens [sum Q_b, hidden].  caches[l]: layer l's cache with the context
        rows in place and room behind them; the query's K/V are written there.  scores_out: fp32 [n_layers, sum T_c]
        or None; when given, row l receives the context scores of layer l from this very pass.  Where scores_out is one matrix and
        weights and caches are lists (or tuples) whose layers have memory of their own, they are computed for up to eight layers at once,
        behind the last of them: the context rows stay as they are until the call's work is done.  A cache that
        several layers share, or that another kind of sequence hands out, is scored before the next layer is asked for.
        Returns the hidden rows after the last layer."""
        rec = self._rec(events)
        h = h0
        group, keep = 1, self.q_kept is not None and scores_out is not None
        for l, w in enumerate(weights):
            h_out = self.h[l % 2]
            cache = caches[l]
            raw = scores_out[l] if scores_out is not None else None
            q, lse = (self.q_kept[l % group], self.lse_kept[l % group]) if keep else (self.q, self.lse)

            def attend():
                nonlocal group
                if l == 0 and keep:                     # (10 us of a host that has three launches ahead of it by now)
                    group = self._score_group(weights, caches, scores_out, events, taps)
                B.relaxkv_query_prefill_attention(self.shape_prefill, cache, q, self.o, lse, None if group > 1 else raw, self.workspace)
            self._block(l, w, cache, h, self.x, self.a, q, self.k, self.v, self.o, self.gu, self.m, h_out,
                        self.q_pos, self.q_cu, self.q_lens, self.shape_ext, attend, rec)
            if group > 1 and (l % group == group - 1 or l == len(weights) - 1):
                l0, n = l - l % group, l % group + 1
                rec("scores", lambda: B.relaxkv_score_select(
                    self.shape_prefill, [self.q_kept[i] for i in range(n)], caches[l0:l + 1], [1] * len(self.ctx_lens),
                    scores_out[l0:l + 1], None, self.workspace, row_lse_layers=[self.lse_kept[i] for i in range(n)]))
            if taps is not None:
                taps.append((h.clone(), h_out.clone()))
            h = h_out
        return h

    def _score_group(self, weights, caches, scores_out, events, taps) -> int:
        """Layers that are scored by one launch (1: each in its own).  More than one need rows of scores_out one behind the other, as a call over
        several layers writes them, and keys that are still there when the last of them has run: nothing of the caller's runs between two
        layers (a generator, a sequence or a list of its own making may fill the next layer's cache then), and no two layers share a byte."""
        if (not isinstance(scores_out, torch.Tensor) or scores_out.dtype != torch.float32 or scores_out.dim() != 2
                or scores_out.shape[1] != sum(self.ctx_lens) or not scores_out.is_contiguous()):
            return 1
        if (any(type(x) not in (list, tuple) for x in (weights, caches)) or any(type(x) not in (list, type(None)) for x in (events, taps))
                or len(caches) < len(weights)):
            return 1
        spans = []
        for c in caches[:len(weights)]:
            v = c.c                                     # (v.v is None for a view without values: refused by the layer's own calls)
            n = 2 * ((c.k.shape[0] - 1) * v.token_stride + (self.Hkv - 1) * v.head_stride + self.D)
            spans += {(v.k, v.k + n), (v.v or 0, (v.v or 0) + n)}          # (one, where K and V are one tensor)
        spans.sort()
        return self.q_kept.shape[0] if all(a[1] <= b[0] for a, b in zip(spans, spans[1:])) else 1

    def decode(self, h_tok: torch.Tensor, weights: List[Dict[str, torch.Tensor]], caches: List[B.CacheView], step: int = 0,
               events: Optional[list] = None) -> torch.Tensor:
        """One decode step: h_tok [n_req, hidden] = the new token's input representation per request; its position is
        T_c + Q_b + step.  Appends its K/V to the caches and returns the hidden row after the last layer."""
        rec = self._rec(events)
        nb = len(self.ctx_lens)
        pos = self.decode_positions(step)
        h = h_tok
        for l, w in enumerate(weights):
            h_out = self.dh[l % 2]

            def attend():
                B.relaxkv_cache_attention(self.shape_dec, caches[l], self.dq, pos, self.d_cu, [1] * nb, self.do, self.workspace)
            self._block(l, w, caches[l], h, self.dx, self.da, self.dq, self.dk, self.dv, self.do, self.dgu, self.dm, h_out,
                        pos, self.d_cu, [1] * nb, self.shape_dec, attend, rec)
            h = h_out
        return h

    def output_head(self, h: torch.Tensor, final_norm: torch.Tensor, w_head: torch.Tensor, logits: torch.Tensor,
                    rows: Optional[torch.Tensor] = None, events: Optional[list] = None) -> torch.Tensor:
        """Final RMSNorm and the output projection of one row per request (by default the last query token's):
        logits [n_req, vocab]."""
        rec = self._rec(events)
        nb = len(self.ctx_lens)
        last = h if h.shape[0] == nb else h.index_select(0, self.last_rows if rows is None else rows)
        rec("head", lambda: (B.relaxkv_rmsnorm(last, final_norm, self.dx, self.blk.eps),
                             B.relaxkv_linear(self.dx, w_head, logits)))
        return logits
