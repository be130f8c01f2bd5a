"""The work a program has this library do, as measurable cases: what Algorithm 1 and the time-to-first-token region around
it consist of, over the model geometries, context lengths, batch shapes and options of this repository's workloads.

Five kinds of pass, each through the public Python entry points:

  score    `RepairSession.score_select` + `build_active_sets`: query-to-context scores of every layer, anchors, schedule
  repair   `relaxkv_select_topk` on given scores, schedule, then per layer sparse-context attention and cache update, with
           the model's projections done elsewhere (fresh Q/K/V rows are in hand)
  blocks   the same schedule, then `LayerLoop.run`: the repair loop with the block work of the active rows
  prefill  `QueryPass.prefill` with the context scores taken from the pass, and the output head of the last row
  decode   `QueryPass.decode` of one token per request and the output head

Every pass leaves its inputs as they were (the cache update writes the same rows again), so it can be repeated.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_33503_b200 import binding as B
from paper_2609_33503_b200 import inputs
from paper_2609_33503_b200.layer_loop import LayerLoop
from paper_2609_33503_b200.pipeline import RepairSession
from paper_2609_33503_b200.query_pass import QueryPass

# head geometry and block sizes: the two model shapes of the benchmark, the decode tests' small model and the tiny workload
LLAMA8B = dict(heads=32, kv_heads=8, head_dim=128, hidden=4096, inter=14336, theta=5.0e5, eps=1.0e-5, qk_norm=False, vocab=128256)
QWEN14B = dict(heads=40, kv_heads=8, head_dim=128, hidden=5120, inter=17408, theta=1.0e6, eps=1.0e-6, qk_norm=True, vocab=151936)
SMALL = dict(heads=8, kv_heads=2, head_dim=128, hidden=2048, inter=4096, theta=1.0e6, eps=1.0e-6, qk_norm=True, vocab=32000)
TINY = dict(heads=4, kv_heads=1, head_dim=64, hidden=256, inter=512, theta=1.0e4, eps=1.0e-5, qk_norm=False, vocab=4096)


def _case(kind, geometry, layers, ctx, query, *, name=None, ratio=0.15, context="union", layout="token", graph=False):
    """ctx, query: tokens per request.  context: "union" (the method) or "full" (the Full-Prefix Control).  layout: which of
    the cache's token and head dimensions is outer.  graph: the program replays the pass from a captured CUDA graph."""
    c = dict(kind=kind, layers=layers, ctx=",".join(map(str, ctx)), query=",".join(map(str, query)), ratio=ratio,
             context=context, layout=layout, graph=graph, **geometry)
    if kind in ("score", "repair"):          # no block work, no output head
        for key in ("hidden", "inter", "theta", "eps", "qk_norm", "vocab"):
            del c[key]
    elif kind == "blocks":
        del c["vocab"]
    return dict(name=name, **c) if name else c


def listed():
    ragged_query = (32, 256, 97, 128, 45, 200, 64, 151)
    return [
        # one layer, 1K context: the smallest call, all launch and host latency
        _case("repair", TINY, 1, [1024], [32], name="repair_1k_tiny"),
        # one 16K layer repaired by itself, 15 % of the tokens
        _case("repair", LLAMA8B, 1, [16384], [64], name="repair_16k_layer"),
        # a whole 32-layer model at 8K, the cache stored head-major (the layout of common inference stacks)
        _case("repair", LLAMA8B, 32, [8192], [64], name="repair_8k_stack", layout="head"),
        # 32K context, twelve layers of the larger model: the ordinary long-context request
        _case("repair", QWEN14B, 12, [32768], [128], name="repair_32k_stack"),
        # a serving batch of eight requests of 8K to 64K tokens in each call
        _case("repair", QWEN14B, 4, inputs.RAGGED_CTX, ragged_query, name="repair_ragged8"),
        # scoring alone: one 16K layer, and all 40 layers of a 32K request in one call
        _case("score", LLAMA8B, 1, [16384], [64], name="score_16k_layer"),
        _case("score", QWEN14B, 40, [32768], [128], name="score_32k_stack"),
        # the query's own forward pass with scores: launched call by call at a ragged length, and replayed from a graph
        _case("prefill", LLAMA8B, 8, [8000], [57], name="prefill_8k"),
        _case("prefill", QWEN14B, 12, [32768], [128], name="prefill_32k", graph=True),
        # one decode step: a small batch launched call by call, and one long-context request from a graph
        _case("decode", LLAMA8B, 16, [8192, 4100, 6001, 2047], [64, 40, 12, 1], name="decode_batch4"),
        _case("decode", QWEN14B, 12, [32768], [128], name="decode_32k", graph=True),
        # the repair loop with block work, where the projections and the MLP take most of the time
        _case("blocks", LLAMA8B, 6, [8192], [64], name="blocks_8k"),
    ]


def _ints(text):
    return [int(x) for x in text.split(",")]


def _cost(c):
    """Rough seconds of a pass, to keep drawn cases below the largest listed one."""
    ctx, query, L = _ints(c["ctx"]), _ints(c["query"]), c["layers"]
    H, D = c["heads"], c["head_dim"]
    params = c["hidden"] * (2 * H + 2 * c["kv_heads"]) * D + 3 * c["hidden"] * c["inter"] if "hidden" in c else 0
    if c["kind"] == "score":
        return sum(4.0 * H * q * t * D for t, q in zip(ctx, query)) * L / 6e14
    if c["kind"] in ("repair", "blocks"):
        pair = 0.5 if c["context"] == "full" else 0.3
        return L * (sum(4.0 * D * H * pair * t * t for t in ctx) / 1e15 + 2.0 * params * 0.5 * sum(ctx) / 1.2e15)
    rows = sum(query) if c["kind"] == "prefill" else len(ctx)
    return L * (2.0 * params / 5e12 + 2.0 * params * rows / 1.2e15 + sum(ctx) * c["kv_heads"] * D * 4 / 4e12)


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["repair", "repair", "score", "prefill", "decode", "blocks"])
    geometry = rng.choice([TINY, SMALL, LLAMA8B, LLAMA8B, QWEN14B, QWEN14B])
    n_req = 1 if rng.random() < 0.5 else rng.randint(2, 8)
    ctx = [spread(512, 65536 if n_req == 1 else 32768) for _ in range(n_req)]
    query = [spread(1, 256) for _ in range(n_req)]
    layers = {"repair": spread(1, 32), "score": spread(1, 40), "blocks": rng.randint(1, 6)}.get(kind, rng.randint(2, 12))
    # a query pass of a batch brings a few hundred rows at most, as the workloads' batches do
    if kind == "prefill":
        query = [max(1, q // n_req) for q in query]
    c = _case(kind, geometry, layers, ctx, query, ratio=round(rng.uniform(0.05, 0.30), 3),
              context="full" if kind == "repair" and rng.random() < 0.25 else "union",
              layout=rng.choice(["token", "token", "head"]), graph=kind in ("prefill", "decode") and rng.random() < 0.5)
    most = max(_cost(x) for x in listed())
    # the state: two caches, fresh rows and outputs of every layer, or the rows of the block work
    rows_limit = {"repair": 400_000, "score": 1_400_000, "blocks": 70_000}.get(kind, 900_000)
    while _cost(c) > most or sum(_ints(c["ctx"])) * (1 if kind == "blocks" else c["layers"]) > rows_limit:
        if c["layers"] > 2 and rng.random() < 0.5:
            c["layers"] -= max(1, c["layers"] // 4)
        else:
            c["ctx"] = ",".join(str(max(512, int(0.8 * t))) for t in _ints(c["ctx"]))
    return c


# ---- inputs -----------------------------------------------------------------------------------------------------------

def _scores(c, seed, device):
    """Context scores of every layer [layers, sum T_c]: positive, summing to one per request and layer, log-normal, with a
    per-request warm set (78 % of the tokens, half of them warm in the first half of the layers only), as in the calibrated
    workloads: the layers' anchors overlap, the union stays below the context and active tokens fall away mid-stack.  The
    seed places the tokens; how many are selected does not depend on it."""
    L, out = c["layers"], []
    for b, t in enumerate(_ints(c["ctx"])):
        g = torch.Generator(device=device).manual_seed(7001 + b)
        warm = torch.rand(t, generator=g, device=device) < 0.78
        early = torch.rand(t, generator=g, device=device) < 0.5
        first = (torch.arange(L, device=device) < (L + 1) // 2)[:, None]
        z = 0.5 * torch.randn(L, t, generator=g, device=device) + 1.0 * (warm & (first | ~early)).float()
        place = torch.randperm(t, generator=g.manual_seed(seed * 1009 + b), device=device)
        out.append(torch.softmax(z, dim=1)[:, place])
    return torch.cat(out, dim=1).contiguous()


def _normal(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.bfloat16)


def _caches(c, rows, seed):
    """K and V of every layer [layers, rows, H_kv, D] ~ N(0,1) (a view of head-major storage where the case says so)."""
    L, Hkv, D = c["layers"], c["kv_heads"], c["head_dim"]
    kv = []
    for n in range(2):
        if c["layout"] == "head":
            kv.append(_normal((L, Hkv, rows, D), seed * 1009 + 31 + n).transpose(1, 2))
        else:
            kv.append(_normal((L, rows, Hkv, D), seed * 1009 + 31 + n))
    return kv


def _offsets(lens):
    return [sum(lens[:b]) for b in range(len(lens))]


def _workload(c, seed):
    return inputs.Workload("case", c["layers"], c["heads"], c["kv_heads"], c["head_dim"], 512, tuple(_ints(c["ctx"])),
                           tuple(_ints(c["query"])), c["ratio"], base_seed=1_000_000 * (seed % 1_000_003), variant="calibrated",
                           warm_seed=12345 + seed)


def _block(c):
    return inputs.BlockShape(hidden=c["hidden"], inter=c["inter"], rope_theta=c["theta"], eps=c["eps"], qk_norm=c["qk_norm"])


def _weights(c, seed):
    """Block weights of every layer, in the layouts the passes read (stacked once, when a program loads its weights)."""
    out = []
    for l in range(c["layers"]):
        w = inputs.block_weights(_workload(c, seed), _block(c), l, "cuda")
        w["w_qkv"] = B.stack_qkv(w.pop("wq"), w.pop("wk"), w.pop("wv"))
        w["w_gate_up_tiled"] = B.tile_gate_up(w.pop("w_gate_up"))
        out.append(w)
    return out


def _anchor_counts(c):
    return [B.relaxkv_anchor_count(t, c["ratio"]) for t in _ints(c["ctx"])]


def _session(c, **kw):
    return RepairSession(c["heads"], c["kv_heads"], c["head_dim"], _ints(c["ctx"]), _ints(c["query"]), c["layers"],
                         _anchor_counts(c), **kw)


def prepare(case, seed):
    c, ctx, query = case, _ints(case["ctx"]), _ints(case["query"])
    L, H, Hkv, D, kind = c["layers"], c["heads"], c["kv_heads"], c["head_dim"], c["kind"]
    st = {"case": c, "layers": L}
    if kind == "score":
        w = _workload(c, seed)
        st["session"] = _session(c, want_norm=True)
        st["q"], st["views"] = [], []
        for l in range(L):
            parts = [inputs.layer_qkv(w, l, b, "cuda")[:2] for b in range(len(ctx))]
            st["q"].append(torch.cat([p[0] for p in parts]))
            k = torch.cat([p[1] for p in parts])
            if c["layout"] == "head":
                k = k.transpose(0, 1).contiguous().transpose(0, 1)
            st["views"].append(B.CacheView(k, None, _offsets(ctx)))
        return st
    if kind in ("repair", "blocks"):
        s = st["session"] = _session(c)
        st["scores"] = _scores(c, seed, "cuda")
        st["k"], st["v"] = _caches(c, sum(ctx), seed)
        st["views"] = [B.CacheView(st["k"][l], st["v"][l], _offsets(ctx)) for l in range(L)]
        rows = s.cap_u
        if kind == "repair":
            st["mode"] = B.CTX_FULL_PREFIX if c["context"] == "full" else B.CTX_UNION
            st["fresh"] = [(_normal((rows, H, D), seed * 1009 + 100 + l), _normal((rows, Hkv, D), seed * 1009 + 200 + l),
                            _normal((rows, Hkv, D), seed * 1009 + 300 + l)) for l in range(L)]
            st["out"] = [torch.empty(rows, H, D, device="cuda", dtype=torch.bfloat16) for _ in range(L)]
        else:
            st["weights"] = _weights(c, seed)
            st["embeddings"] = [_normal((t, c["hidden"]), seed * 1009 + 400 + b) for b, t in enumerate(ctx)]
            st["loop"] = LayerLoop(s, _block(c), rows)
        return st
    # prefill / decode: room behind every request's context for its query and one decoded token
    room = [t + q + 1 for t, q in zip(ctx, query)]
    st["k"], st["v"] = _caches(c, sum(room), seed)
    st["views"] = [B.CacheView(st["k"][l], st["v"][l], _offsets(room)) for l in range(L)]
    st["weights"] = _weights(c, seed)
    qp = st["pass"] = QueryPass(H, Hkv, D, ctx, query, _block(c))
    st["x"] = _normal((sum(query) if kind == "prefill" else len(ctx), c["hidden"]), seed * 1009 + 500)
    st["final_norm"] = 1 + 0.1 * _normal((c["hidden"],), seed * 1009 + 501)
    st["w_head"] = _normal((c["vocab"], c["hidden"]), seed * 1009 + 502) * c["hidden"] ** -0.5
    st["logits"] = torch.empty(len(ctx), c["vocab"], device="cuda", dtype=torch.bfloat16)
    n_new = query if kind == "prefill" else [1] * len(ctx)
    at = [o + t + (0 if kind == "prefill" else q) for o, t, q in zip(_offsets(room), ctx, query)]
    st["appended"] = [x[:, a:a + n] for x in (st["k"], st["v"]) for a, n in zip(at, n_new)]
    if kind == "prefill":
        st["raw"] = torch.empty(L, sum(ctx), device="cuda", dtype=torch.float32)
    else:
        qp.decode_positions(0)
    if c["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _query_side(st)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                st["hidden"] = _query_side(st)
        torch.cuda.current_stream().wait_stream(side)
        st["graph"] = graph
    return st


# ---- one pass -----------------------------------------------------------------------------------------------------------

def _query_side(st):
    qp = st["pass"]
    if st["case"]["kind"] == "prefill":
        h = qp.prefill(st["x"], st["weights"], st["views"], scores_out=st["raw"])
    else:
        h = qp.decode(st["x"], st["weights"], st["views"], step=0)
    qp.output_head(h, st["final_norm"], st["w_head"], st["logits"])
    return h


def run(st):
    kind = st["case"]["kind"]
    if kind == "score":
        s = st["session"]
        s.score_select(st["q"], st["views"])
        s.build_active_sets()
        return {"raw": s.raw, "norm": s.norm, "highest_layer": s.highest_layer}
    if kind in ("prefill", "decode"):
        if "graph" in st:
            st["graph"].replay()
            h = st["hidden"]
        else:
            h = _query_side(st)
        out = {"logits": st["logits"], "hidden": h, "appended": st["appended"]}
        return dict(out, raw=st["raw"]) if kind == "prefill" else out
    s = st["session"]
    B.relaxkv_select_topk(s.shape, st["layers"], s.k, st["scores"], s.anchors)
    s.build_active_sets()
    n_u, n_r = s.counts()
    out = {"anchors": s.anchors, "highest_layer": s.highest_layer, "u_pos": s.u_pos[:sum(n_u)], "u_rank": s.u_rank,
           "r_rank": s.r_rank[:sum(map(sum, n_r))], "r_cu": s.r_cu, "k": st["k"], "v": st["v"]}
    if kind == "repair":
        out["out"] = []
        for l in range(st["layers"]):
            n = sum(n_r[l])
            q, k, v = (x[:n] for x in st["fresh"][l])
            o = st["out"][l][:n]
            s.attention(l, st["views"][l], q, k, v, o, n_r[l], n_u, mode=st["mode"])
            s.scatter(l, st["views"][l], k, v, n_r[l])
            out["out"].append(o)
        return out
    at, rows = 0, []
    for n, table in zip(n_u, st["embeddings"]):
        rows.append(table.index_select(0, s.u_pos[at:at + n]))
        at += n
    out["hidden"] = st["loop"].run(rows[0] if len(rows) == 1 else torch.cat(rows), st["weights"], st["views"])
    return out


# ---- what a pass cannot do without ----------------------------------------------------------------------------------------

def _sets(c):
    """Per layer, summed over the requests: (targets, context rows, edges), for the scores of one seed."""
    L, at, k = c["layers"], 0, _anchor_counts(c)
    scores = _scores(c, 1, "cpu").numpy()
    n_r, n_u, edges = np.zeros(L), 0, np.zeros(L)
    for b, t in enumerate(_ints(c["ctx"])):
        high = np.full(t, -1)
        for l in range(L):
            high[np.argpartition(-scores[l, at:at + t], k[b] - 1)[:k[b]]] = l
        at += t
        u = np.flatnonzero(high >= 0)
        n_u += t if c["context"] == "full" else len(u)
        limit = u + 1 if c["context"] == "full" else np.arange(len(u)) + 1
        for l in range(L):
            n_r[l] += (high[u] >= l).sum()
            edges[l] += limit[high[u] >= l].sum()
    return n_r, n_u, edges


def work(case):
    c, ctx, query = case, _ints(case["ctx"]), _ints(case["query"])
    L, H, Hkv, D, T = c["layers"], c["heads"], c["kv_heads"], c["head_dim"], sum(ctx)
    kv_row, q_row = 4 * Hkv * D, 2 * H * D                                        # bytes of a token's K and V, of its Q
    if c["kind"] == "score":
        return {"bytes": L * (T * kv_row / 2 + sum(query) * q_row + 8 * T) + 4 * T,
                "flops": L * sum(2.0 * H * D * q * t for t, q in zip(ctx, query))}
    layer_weights = c["hidden"] * (2 * H + 2 * Hkv) * D + 3 * c["hidden"] * c["inter"] if "hidden" in c else 0
    if c["kind"] in ("repair", "blocks"):
        n_r, n_u, edges = _sets(c)
        k = sum(_anchor_counts(c))
        lists = 4 * L * (T + k) + 8 * T + 4 * n_u + 4 * n_r.sum()
        flops = 4.0 * D * H * edges.sum()
        if c["kind"] == "repair":    # Q in, output out, fresh K/V in and to the cache, cached K/V of the context's other rows
            per_layer = n_r * (2 * q_row + 2 * kv_row) + (n_u - n_r) * kv_row
            return {"bytes": lists + per_layer.sum(), "flops": flops}
        per_layer = n_r * kv_row + (n_u - n_r) * kv_row + 2 * layer_weights
        return {"bytes": lists + per_layer.sum() + 4 * n_u * c["hidden"], "flops": flops + 2.0 * layer_weights * n_r.sum()}
    rows = sum(query) if c["kind"] == "prefill" else len(ctx)
    per_layer = 2 * layer_weights + T * kv_row + rows * kv_row
    edges = sum(q * t + q * (q + 1) / 2 for t, q in zip(ctx, query)) if c["kind"] == "prefill" else sum(
        t + q + 1 for t, q in zip(ctx, query))
    head = c["vocab"] * c["hidden"]
    raw = 4 * L * T if c["kind"] == "prefill" else 0
    return {"bytes": L * per_layer + 2 * head + 2 * len(ctx) * c["vocab"] + raw,
            "flops": L * (2.0 * layer_weights * rows + 4.0 * D * H * edges) + 2.0 * head * len(ctx)}


def tolerance(case):
    """About four times what each kind differs by from the same pass in 64 bits: scores 2e-7 (fp32 sums and exponentials; an
    anchor may change where two scores agree to the last bits), one attention 2.1e-3 (probabilities and results rounded to
    bf16; 0.03 in single values), chains of 6 to 12 layers 8e-3 to 1.3e-2 (0.06 in single values)."""
    if case["kind"] == "score":
        return {"rel": 2e-6, "max": 8e-6, "differ": 4e-3}
    if case["kind"] == "repair":
        return {"rel": 8e-3, "max": 0.12, "differ": 0.0}
    return {"rel": 2.5e-2, "max": 0.25, "differ": 0.0}
