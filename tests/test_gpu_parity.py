"""GPU parity: every C-ABI call against the fp64 CPU oracle on the same seeded bits.

Tolerances (bf16 inputs, fp32 accumulation, P rounded to bf16 before P*V):
  attention outputs  max-abs <= 2e-2, mean-abs <= 2e-3
  raw scores         |gpu - ref| <= 1e-3 * ref + 1e-6 / T_c ;  normalised scores abs <= 1e-3
  anchors            bit-exact when scores are fed in exactly; otherwise exact outside a 1e-3
                     relative band around the k-th score
  sets, gather, scatter: bit-exact
"""
import numpy as np
import pytest
import torch

from oracle import relaxkv_oracle as orc
from paper_2609_33503_b200 import inputs
from tests.harness import Case, attention_errors, bf16_to_f64, check_anchor_band

pytestmark = pytest.mark.gpu

MAX_ABS, MEAN_ABS = 2e-2, 2e-3


def B():
    from paper_2609_33503_b200 import binding
    return binding


def assert_status_ok():
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (B().status_string(st), detail)


def small_llama(n_layers=2, ctx=(2048,), q=(48,)):
    return inputs.scaled_down(inputs.llama8b_16k(), ctx, q, n_layers=n_layers, chunk=256)


def small_qwen(n_layers=3, ctx=(1536,), q=(40,)):
    return inputs.scaled_down(inputs.qwen14b_32k("calibrated"), ctx, q, n_layers=n_layers, chunk=128)


def small_ragged():
    return inputs.scaled_down(inputs.qwen14b_32k("calibrated"), (640, 1280, 2176), (17, 33, 64), n_layers=2, chunk=128)


WORKLOADS = {
    "tiny": inputs.tiny,
    "llama_small": small_llama,
    "qwen_small": small_qwen,
    "ragged_small": small_ragged,
}


@pytest.fixture(scope="module", params=list(WORKLOADS))
def case(request):
    return Case(WORKLOADS[request.param]())


# ------------------------------------------------------------------------- selection ----

def test_scores_and_anchors(case):
    w = case.w
    s = case.make_session(want_norm=True)
    s.score_select(case.q_layers, case.cache_views())
    assert_status_ok()
    raw = s.raw.cpu().numpy().astype(np.float64)
    norm = s.norm.cpu().numpy().astype(np.float64)
    anchors = s.anchors.cpu().numpy()
    for l in range(w.n_layers):
        for b in range(w.n_req):
            T = w.ctx_lens[b]
            ref = case.raw[(l, b)]
            got = raw[l, case.ctx_cu[b]:case.ctx_cu[b + 1]]
            assert np.all(np.abs(got - ref) <= 1e-3 * ref + 1e-6 / T), np.abs(got / ref - 1).max()
            assert abs(got.sum() - 1.0) < 1e-3
            np.testing.assert_allclose(norm[l, case.ctx_cu[b]:case.ctx_cu[b + 1]], orc.minmax(ref), atol=1e-3)
            check_anchor_band(ref, case.k[b], anchors[l, case.k_cu[b]:case.k_cu[b + 1]])


def test_scores_with_supplied_lse(case):
    """Supplying the rows' log-normalisers skips the statistics pass and gives the same scores."""
    w = case.w
    s = case.make_session()
    lses = []
    for l in range(w.n_layers):
        per_req = [orc.row_lse(case.req_q(l, b), case.req_k(l, b), case.scale) for b in range(w.n_req)]
        lses.append(torch.from_numpy(np.concatenate(per_req, axis=1).astype(np.float32)).contiguous().to(case.device))
    s.score_select(case.q_layers, case.cache_views(), row_lse_layers=lses)
    assert_status_ok()
    raw = s.raw.cpu().numpy().astype(np.float64)
    for l in range(w.n_layers):
        for b in range(w.n_req):
            ref = case.raw[(l, b)]
            got = raw[l, case.ctx_cu[b]:case.ctx_cu[b + 1]]
            assert np.all(np.abs(got - ref) <= 1e-3 * ref + 1e-6 / w.ctx_lens[b])


def test_select_exact_on_given_scores(case):
    """Oracle scores rounded to fp32 go in; anchors must match the oracle's top-k of those very
    values bit for bit (ties included: a block of equal scores is planted)."""
    w = case.w
    nb, L = w.n_req, w.n_layers
    shape = case.make_session().shape
    raw32 = np.zeros((L, int(case.ctx_cu[-1])), dtype=np.float32)
    for l in range(L):
        for b in range(nb):
            r = case.raw[(l, b)].astype(np.float32)
            kth = np.sort(r)[::-1][case.k[b] - 1]
            idx = np.argsort(np.abs(r - kth))[:9]        # make 9 scores tie with the k-th one
            r[idx] = kth
            raw32[l, case.ctx_cu[b]:case.ctx_cu[b + 1]] = r
    d_raw = torch.from_numpy(raw32).to(case.device)
    d_anchor = torch.full((L, int(case.k_cu[-1])), -1, dtype=torch.int32, device=case.device)
    d_norm = torch.empty_like(d_raw)
    B().relaxkv_select_topk(shape, L, case.k, d_raw, d_anchor, norm_scores_out=d_norm)
    assert_status_ok()
    got = d_anchor.cpu().numpy()
    for l in range(L):
        for b in range(nb):
            seg = raw32[l, case.ctx_cu[b]:case.ctx_cu[b + 1]].astype(np.float64)
            np.testing.assert_array_equal(got[l, case.k_cu[b]:case.k_cu[b + 1]], orc.topk(seg, case.k[b]))
            np.testing.assert_allclose(d_norm[l, case.ctx_cu[b]:case.ctx_cu[b + 1]].cpu().numpy(), orc.minmax(seg),
                                       atol=2e-6)


def test_active_sets_bitexact(case):
    w = case.w
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    assert_status_ok()
    n_u, n_r = s.counts()
    u_cu = s.u_cu.cpu().numpy()
    r_cu = s.r_cu.cpu().numpy()
    u_pos, u_rank, h = s.u_pos.cpu().numpy(), s.u_rank.cpu().numpy(), s.highest_layer.cpu().numpy()
    r_rank = s.r_rank.cpu().numpy()
    for b in range(w.n_req):
        ref = case.sets[b]
        assert n_u[b] == len(ref.u_pos) == u_cu[b + 1] - u_cu[b]
        np.testing.assert_array_equal(u_pos[u_cu[b]:u_cu[b + 1]], ref.u_pos)
        np.testing.assert_array_equal(u_rank[case.ctx_cu[b]:case.ctx_cu[b + 1]], ref.u_rank)
        np.testing.assert_array_equal(h[case.ctx_cu[b]:case.ctx_cu[b + 1]], ref.h)
        prev = None
        for l in range(w.n_layers):
            i = l * w.n_req + b
            got = r_rank[r_cu[i]:r_cu[i + 1]]
            np.testing.assert_array_equal(got, ref.ranks(l))
            assert n_r[l][b] == len(got)
            if prev is not None:
                assert set(got.tolist()) <= prev                     # monotone across layers
            prev = set(got.tolist())


@pytest.mark.parametrize("ctx", [(1,), (31, 33), (4096,), (4097, 1, 640), (8193, 20000), (16385,), (40000, 7), (196609,)])
def test_selection_and_schedule_at_slice_edges(ctx):
    """Top-k, MinMax and the schedule where the slices of a segment (1, 2, 4 or 8 blocks), their warps' runs and the keys kept in
    shared memory (196609 is past them) begin and end: bit-exact on scores with ties, both signs, zeros and infinities."""
    from paper_2609_33503_b200.pipeline import RepairSession
    rng = np.random.default_rng(sum(ctx))
    L, nb = 3, len(ctx)
    cu = np.concatenate([[0], np.cumsum(ctx)])
    raw = np.empty((L, cu[-1]), dtype=np.float32)
    raw[0] = np.exp(rng.standard_normal(cu[-1])) / cu[-1]
    raw[1] = np.round(rng.standard_normal(cu[-1]) * 3) / 4                 # many ties, both signs and zeros
    raw[2] = rng.standard_normal(cu[-1])
    raw[2, ::3] = -np.inf
    raw[2, ::5] = np.inf
    for k in ([1] * nb, [max(1, round(0.15 * t)) for t in ctx], list(ctx)):
        s = RepairSession(8, 2, 128, ctx, [1] * nb, L, k)
        d_raw = torch.from_numpy(raw).cuda()
        d_norm = torch.empty_like(d_raw)
        B().relaxkv_select_topk(s.shape, L, s.k, d_raw, s.anchors, norm_scores_out=d_norm)
        s.build_active_sets()
        n_u, n_r = s.counts()
        assert_status_ok()
        anchors, norm = s.anchors.cpu().numpy(), d_norm.cpu().numpy()
        k_cu = np.concatenate([[0], np.cumsum(k)])
        u_cu, r_cu, r_rank = s.u_cu.cpu().numpy(), s.r_cu.cpu().numpy(), s.r_rank.cpu().numpy()
        for b in range(nb):
            seg = slice(cu[b], cu[b + 1])
            want = [orc.topk(raw[l, seg].astype(np.float64), k[b]) for l in range(L)]
            for l in range(L):
                np.testing.assert_array_equal(anchors[l, k_cu[b]:k_cu[b + 1]], want[l])
                if l < 2:                                                  # the same fp32 arithmetic: the same bits
                    x = raw[l, seg]
                    rng_x = x.max() - x.min()
                    np.testing.assert_array_equal(norm[l, seg], (x - x.min()) / rng_x if rng_x > 0 else np.zeros_like(x))
            ref = orc.active_sets(np.stack(want), ctx[b])
            assert n_u[b] == len(ref.u_pos) == u_cu[b + 1] - u_cu[b]
            np.testing.assert_array_equal(s.u_pos[u_cu[b]:u_cu[b + 1]].cpu().numpy(), ref.u_pos)
            np.testing.assert_array_equal(s.u_rank[cu[b]:cu[b + 1]].cpu().numpy(), ref.u_rank)
            for l in range(L):
                got = r_rank[r_cu[l * nb + b]:r_cu[l * nb + b + 1]]
                assert n_r[l][b] == len(got)
                np.testing.assert_array_equal(got, ref.ranks(l))


@pytest.mark.parametrize("ctx,L", [((8192, 100), 70), ((8193,), 32), ((8193, 5), 32), ((30000,), 33), ((49153,), 9), ((49153, 1), 5), ((24577,), 70),
                                   ((98305,), 12)])
def test_selection_by_segments_of_a_call(ctx, L):
    """The slices of a segment follow from the longest one and from how many segments run at once (32 of four slices, 64 of two): on
    both sides of each limit the anchors are the oracle's, with ties, bit for bit."""
    rng = np.random.default_rng(L + sum(ctx))
    cu = np.concatenate([[0], np.cumsum(ctx)])
    k = [max(1, round(0.15 * t)) for t in ctx]
    k_cu = np.concatenate([[0], np.cumsum(k)])
    raw = (np.round(rng.standard_normal((L, cu[-1])) * 200) / 200).astype(np.float32)
    anchors = torch.full((L, k_cu[-1]), -1, dtype=torch.int32, device="cuda")
    B().relaxkv_select_topk(B().Shape(8, 2, 128, list(ctx)), L, k, torch.from_numpy(raw).cuda(), anchors)
    assert_status_ok()
    got = anchors.cpu().numpy()
    for l in range(L):
        for b in range(len(ctx)):
            np.testing.assert_array_equal(got[l, k_cu[b]:k_cu[b + 1]], orc.topk(raw[l, cu[b]:cu[b + 1]].astype(np.float64), k[b]))


@pytest.mark.parametrize("ctx,L", [((1,) + tuple(range(33, 96)), 6), ((1024,) * 64, 40), ((4097,) * 3 + (31, 32, 1), 40), ((65536, 640), 60),
                                   ((32768,), 40), ((32769, 5), 12), ((100001,), 6), ((70000, 4096, 1, 16385), 3)])
def test_schedule_by_the_blocks_per_list(ctx, L):
    """Schedules of few long lists to many short ones (one to eight blocks share a list): every output bit-exact against the oracle,
    with a sixth of the positions never selected and the anchors of a request's layers overlapping."""
    from paper_2609_33503_b200.pipeline import RepairSession
    rng = np.random.default_rng(len(ctx) * 1000 + L)
    nb, k = len(ctx), [max(1, t // 9) for t in ctx]
    cu = np.concatenate([[0], np.cumsum(ctx)])
    want = [np.stack([np.sort(rng.choice(max(1, t - t // 6), size=kb, replace=False)) for _ in range(L)]).astype(np.int32) for t, kb in zip(ctx, k)]
    s = RepairSession(8, 2, 128, ctx, [1] * nb, L, k)
    for t in (s.highest_layer, s.u_pos, s.u_cu, s.u_rank, s.r_rank, s.r_cu, s.counts_pinned):
        t.fill_(-7)
    s.build_active_sets(torch.from_numpy(np.concatenate(want, axis=1)).cuda())
    n_u, n_r = s.counts()
    assert_status_ok()
    u_cu, r_cu, u_pos, u_rank, r_rank = (t.cpu().numpy() for t in (s.u_cu, s.r_cu, s.u_pos, s.u_rank, s.r_rank))
    assert u_cu[0] == r_cu[0] == 0
    for b in range(nb):
        ref = orc.active_sets(want[b], ctx[b])
        assert n_u[b] == len(ref.u_pos) == u_cu[b + 1] - u_cu[b]
        np.testing.assert_array_equal(u_pos[u_cu[b]:u_cu[b + 1]], ref.u_pos)
        np.testing.assert_array_equal(u_rank[cu[b]:cu[b + 1]], ref.u_rank)
        for l in range(L):
            got = r_rank[r_cu[l * nb + b]:r_cu[l * nb + b + 1]]
            assert n_r[l][b] == len(got)
            np.testing.assert_array_equal(got, ref.ranks(l))


# --------------------------------------------------------------------- gather / scatter ----

@pytest.mark.parametrize("head_major", [False, True])
def test_gather_and_scatter_bitexact(head_major):
    case = Case(small_ragged(), head_major_cache=head_major)
    w = case.w
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    nb = w.n_req
    for l in range(w.n_layers):
        f = case.fresh[l]
        views = case.cache_views()
        for mode in (B().CTX_UNION, B().CTX_FULL_PREFIX):
            rows = (sum(case.max_ctx()) if mode == B().CTX_UNION else int(case.ctx_cu[-1])) + 64
            kc = torch.full((rows, w.n_kv_heads, w.head_dim), 7.0, dtype=torch.bfloat16, device=case.device)
            vc = torch.full_like(kc, 7.0)
            s.gather(l, views[l], f.k_new, f.v_new, case.max_ctx(), kc, vc, mode=mode)
            assert_status_ok()
            kc_b, vc_b = inputs.bf16_bits(kc), inputs.bf16_bits(vc)
            off = 0
            for b in range(nb):
                _, kn, vn = case.fresh_bits(l, b)
                st = case.sets[b]
                if mode == B().CTX_UNION:
                    rk, rv = orc.mix_context(case.req_k(l, b), case.req_v(l, b), kn, vn, st.u_pos, st.ranks(l))
                else:
                    T = w.ctx_lens[b]
                    rk, rv = orc.mix_context(case.req_k(l, b), case.req_v(l, b), kn, vn,
                                             np.arange(T, dtype=np.int32), st.positions(l))
                np.testing.assert_array_equal(kc_b[off:off + len(rk)], rk)
                np.testing.assert_array_equal(vc_b[off:off + len(rv)], rv)
                off += len(rk)
            assert np.all(kc_b[off:off + 64] == 0) and np.all(vc_b[off:off + 64] == 0)     # zero pad rows
        # scatter into a copy of the cache
        k2, v2 = case.k_cache[l].clone(), case.v_cache[l].clone()
        if head_major:
            k2 = case.k_cache[l].permute(1, 0, 2).contiguous().permute(1, 0, 2)
            v2 = case.v_cache[l].permute(1, 0, 2).contiguous().permute(1, 0, 2)
        view2 = B().CacheView(k2, v2, [int(x) for x in case.ctx_cu[:-1]])
        for _ in range(2):                                            # idempotent
            s.scatter(l, view2, f.k_new, f.v_new, case.max_targets(l))
        assert_status_ok()
        k2_b, v2_b = inputs.bf16_bits(k2), inputs.bf16_bits(v2)
        for b in range(nb):
            rk, rv = case.req_k(l, b).copy(), case.req_v(l, b).copy()
            _, kn, vn = case.fresh_bits(l, b)
            orc.scatter(rk, rv, kn, vn, case.sets[b].positions(l))
            np.testing.assert_array_equal(k2_b[case.ctx_cu[b]:case.ctx_cu[b + 1]], rk)
            np.testing.assert_array_equal(v2_b[case.ctx_cu[b]:case.ctx_cu[b + 1]], rv)


# ---------------------------------------------------------------------------- attention ----

def run_attention(case, s, l, mode, simt, use_fresh=True, views=None):
    w = case.w
    f = case.fresh[l]
    out = torch.zeros_like(f.q_new)
    lse = torch.zeros(w.n_q_heads, f.q_new.shape[0], dtype=torch.float32, device=case.device)
    views = views or case.cache_views()
    s.attention(l, views[l], f.q_new, f.k_new if use_fresh else None, f.v_new if use_fresh else None, out,
                case.max_targets(l), case.max_ctx(), mode=mode, lse_out=lse, simt=simt)
    assert_status_ok()
    return out, lse


def check_attention(case, l, out, lse, full_prefix, use_fresh=True):
    f = case.fresh[l]
    worst = (0.0, 0.0)
    for b in range(case.w.n_req):
        lo, hi = f.row_cu[b], f.row_cu[b + 1]
        if hi == lo:
            continue
        ref, ref_lse = case.oracle_attention(l, b, full_prefix=full_prefix, use_fresh_kv=use_fresh)
        mx, mean = attention_errors(out[lo:hi], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (l, b, mx, mean)
        got_lse = lse[:, lo:hi].cpu().numpy().astype(np.float64).T
        np.testing.assert_allclose(got_lse, ref_lse, atol=2e-3, rtol=1e-4)
        worst = (max(worst[0], mx), max(worst[1], mean))
    return worst


@pytest.mark.parametrize("simt", [True, False], ids=["simt", "tcgen05"])
@pytest.mark.parametrize("full_prefix", [False, True], ids=["union", "fullprefix"])
def test_attention_matches_oracle(case, simt, full_prefix):
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    mode = B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION
    for l in range(case.w.n_layers):
        out, lse = run_attention(case, s, l, mode, simt)
        check_attention(case, l, out, lse, full_prefix)


@pytest.mark.parametrize("n_splits", [1, 2, 5, 32])
def test_context_split_matches_oracle(case, n_splits):
    """Few query tiles: the context of every tile pair is split over several blocks and the partial results are
    merged by their log-sum-exp.  Forced here to 1 (never), 2, 5 and 32 splits (more splits than some pairs have
    context tiles: empty splits), in both context modes, against the oracle; the rows past the true target count
    of a loosely bounded call stay untouched."""
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    s.shape.set_tuning(attention_ctx_splits=n_splits)
    try:
        for l in range(case.w.n_layers):
            for full_prefix in (False, True):
                out, lse = run_attention(case, s, l, B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION, simt=False)
                check_attention(case, l, out, lse, full_prefix)
        f = case.fresh[0]
        n = f.q_new.shape[0]
        pad = 7
        q_pad = torch.cat([f.q_new, torch.zeros(pad, *f.q_new.shape[1:], dtype=f.q_new.dtype, device=f.q_new.device)])
        out = torch.full_like(q_pad, 3.0)
        s.attention(0, case.cache_views()[0], q_pad, f.k_new, f.v_new, out, list(case.w.ctx_lens), list(case.w.ctx_lens))
        assert_status_ok()
        assert torch.all(out[n:] == 3.0)
        exact, _ = run_attention(case, s, 0, B().CTX_UNION, simt=False)
        assert torch.equal(out[:n], exact)
    finally:
        s.shape.set_tuning()


@pytest.mark.parametrize("blocks", [1, 3, 0], ids=["one_block", "three_blocks", "one_per_sm"])
def test_persistent_form_matches_oracle_and_the_one_shot_kernel(case, blocks):
    """The persistent form of the attention kernel (one block walks many query-tile pairs, claimed from a counter):
    forced on, with a single block walking every item, with three, and with one per SM; both context modes against
    the oracle, bit-identical to the one-shot kernel, rows past a loosely bounded call's true count untouched."""
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    try:
        for l in range(case.w.n_layers):
            for full_prefix in (False, True):
                mode = B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION
                s.shape.set_tuning(attention_ctx_splits=1, attention_persistent=2)
                ref, ref_lse = run_attention(case, s, l, mode, simt=False)
                s.shape.set_tuning(attention_ctx_splits=1, attention_persistent=1, attention_grid_blocks=blocks)
                out, lse = run_attention(case, s, l, mode, simt=False)
                check_attention(case, l, out, lse, full_prefix)
                assert torch.equal(out, ref) and torch.equal(lse, ref_lse)
        f = case.fresh[0]
        n = f.q_new.shape[0]
        q_pad = torch.cat([f.q_new, torch.zeros(7, *f.q_new.shape[1:], dtype=f.q_new.dtype, device=f.q_new.device)])
        out = torch.full_like(q_pad, 3.0)
        s.attention(0, case.cache_views()[0], q_pad, f.k_new, f.v_new, out, list(case.w.ctx_lens), list(case.w.ctx_lens))
        assert_status_ok()
        assert torch.all(out[n:] == 3.0)
    finally:
        s.shape.set_tuning()


@pytest.mark.parametrize("persistent", [2, 1], ids=["one_shot", "persistent"])
def test_attention_call_replays_from_a_cuda_graph(persistent):
    """Gather + attention captured into a CUDA graph (the persistent form also zeroes its work counter there) and
    replayed twice give the bits of the eager call."""
    case = Case(small_llama())
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    s.shape.set_tuning(attention_ctx_splits=1, attention_persistent=persistent, attention_grid_blocks=2)
    try:
        eager, eager_lse = run_attention(case, s, 0, B().CTX_UNION, simt=False)
        f = case.fresh[0]
        out = torch.zeros_like(f.q_new)
        lse = torch.zeros_like(eager_lse)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side):
            with torch.cuda.graph(g, stream=side):
                s.attention(0, case.cache_views()[0], f.q_new, f.k_new, f.v_new, out, case.max_targets(0), case.max_ctx(),
                            mode=B().CTX_UNION, lse_out=lse)
        torch.cuda.current_stream().wait_stream(side)
        for _ in range(2):
            out.zero_(); lse.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert_status_ok()
            assert torch.equal(out, eager) and torch.equal(lse, eager_lse)
    finally:
        s.shape.set_tuning()


@pytest.mark.parametrize("shape", ["five_heads", "four_heads", "head_dim_64"])
@pytest.mark.parametrize("growth", [3.0, 30.0])
def test_row_maxima_that_grow_along_the_context(shape, growth):
    """Keys that grow along the context: the row maxima outgrow the reference of the tiles before, once or several times per row, so that
    O is rescaled (at 3 a few rows of a warp, at 30 all of them).  One block per tile pair, the persistent form and a context split.  Values at a quarter: a row that one key dominates takes its value, of up
    to 4.5, rounded twice (P and O, 2^-9 each) = 0.018, which is the tolerance itself."""
    w = {"five_heads": inputs.scaled_down(inputs.qwen14b_32k("literal"), (1500,), (5,), n_layers=1, chunk=64),
         "four_heads": small_llama(n_layers=1, ctx=(1300, 700), q=(8, 8)), "head_dim_64": inputs.tiny()}[shape].replace(ratio=0.5)
    case = Case(w)
    f = case.fresh[0]
    n = f.k_new.shape[0]
    ramp = torch.linspace(1.0, growth, n, device=f.k_new.device)[:, None, None]
    f.k_new = (f.k_new.float() * ramp).to(torch.bfloat16)
    f.v_new = (f.v_new.float() * 0.25).to(torch.bfloat16)
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    for tuning in (dict(attention_ctx_splits=1, attention_persistent=2), dict(attention_ctx_splits=1, attention_persistent=1, attention_grid_blocks=3),
                   dict(attention_ctx_splits=2)):
        s.shape.set_tuning(**tuning)
        out, lse = run_attention(case, s, 0, B().CTX_UNION, simt=False)
        check_attention(case, 0, out, lse, False)


def test_row_maxima_that_grow_do_not_cost_the_exponentials_twice():
    """One layer of 8 K tokens (dim 64, where the exponential unit bounds the step) with keys that grow thirtyfold along the context
    against keys that do not.  Rescaling O in most steps costs 9 %; exponentials done again besides cost 56 %: the bound lies between."""
    g = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda n, h: torch.randn(n, h, 64, device="cuda", generator=g).to(torch.bfloat16)
    from paper_2609_33503_b200.pipeline import RepairSession
    n = 6144
    s = RepairSession(32, 8, 64, [8192], [8], 1, [n])
    s.build_active_sets(torch.randperm(8192, device="cuda", generator=g)[:n].sort().values.to(torch.int32).view(1, n).contiguous())
    view = B().CacheView(rnd(8192, 8), rnd(8192, 8), [0])
    q, k, v = rnd(n, 32), rnd(n, 8), rnd(n, 8)
    grown = (k.float() * torch.linspace(1.0, 30.0, n, device="cuda")[:, None, None]).to(torch.bfloat16)
    out = torch.empty_like(q)

    def us(keys, reps=20):
        t = []
        for _ in range(2):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(reps):
                s.attention(0, view, q, keys, v, out, [n], [n])
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]) / reps * 1e3)
        return t[-1]

    ratio = sorted(us(grown) / us(k) for _ in range(7))[3]
    assert_status_ok()
    assert ratio < 1.3, ratio


@pytest.mark.parametrize("kind", [np.int64, np.int32, torch.tensor], ids=["int64", "int32", "tensor"])
def test_a_layer_is_any_integer(kind):
    """The layer of a session's calls may be a numpy or torch integer, as an index of a tensor may."""
    case = Case(small_llama())
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    l = case.w.n_layers - 1
    ref, _ = run_attention(case, s, l, B().CTX_UNION, simt=False)
    f = case.fresh[l]
    out = torch.zeros_like(ref)
    s.attention(kind(l), case.cache_views()[l], f.q_new, f.k_new, f.v_new, out, case.max_targets(l), case.max_ctx())
    s.scatter(kind(l), case.cache_views()[l], f.k_new, f.v_new, case.max_targets(l))
    assert_status_ok()
    assert torch.equal(out, ref)


def test_attention_orders_agree_and_is_deterministic(case):
    """Update-then-attend from the cache equals mix-then-attend (Algorithm 1's order), bit for bit;
    two runs give identical bits."""
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    l = case.w.n_layers - 1
    f = case.fresh[l]
    a, _ = run_attention(case, s, l, B().CTX_UNION, simt=False)
    a2, _ = run_attention(case, s, l, B().CTX_UNION, simt=False)
    assert torch.equal(a, a2)
    k2, v2 = case.k_cache[l].clone(), case.v_cache[l].clone()
    view2 = B().CacheView(k2, v2, [int(x) for x in case.ctx_cu[:-1]])
    s.scatter(l, view2, f.k_new, f.v_new, case.max_targets(l))
    views = list(case.cache_views())
    views[l] = view2
    b_out, _ = run_attention(case, s, l, B().CTX_UNION, simt=False, use_fresh=False, views=views)
    assert torch.equal(a, b_out)


def test_full_ratio_is_dense_causal_attention():
    """Anchor ratio 100 %: every position is an anchor at every layer, so the output must equal plain
    causal attention over the fresh K/V (library SDPA in fp32 on the GPU, fp64 oracle on the CPU)."""
    w = small_llama(n_layers=1, ctx=(700,), q=(8,)).replace(ratio=1.0)
    case = Case(w)
    assert case.k == [700]
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    out, lse = run_attention(case, s, 0, B().CTX_UNION, simt=False)
    check_attention(case, 0, out, lse, False)
    f = case.fresh[0]
    G = w.group
    q = f.q_new.float().permute(1, 0, 2).unsqueeze(0)
    k = f.k_new.float().repeat_interleave(G, dim=1).permute(1, 0, 2).unsqueeze(0)
    v = f.v_new.float().repeat_interleave(G, dim=1).permute(1, 0, 2).unsqueeze(0)
    ref = torch.nn.functional.scaled_dot_product_attention(q, k, v, is_causal=True, scale=case.scale)[0].permute(1, 0, 2)
    d = (out.float() - ref).abs()
    assert d.max().item() <= MAX_ABS and d.mean().item() <= MEAN_ABS


@pytest.mark.parametrize("ctx,q,ratio", [((1,), (1,), 0.15), ((129,), (3,), 0.01), ((257,), (5,), 1.0), ((130, 1, 515), (2, 1, 7), 0.3),
                                         ((1000, 300), (200, 131), 0.15)])
def test_edge_sizes(ctx, q, ratio):
    w = inputs.scaled_down(inputs.qwen14b_32k("literal"), ctx, q, n_layers=2, chunk=64).replace(ratio=ratio)
    case = Case(w)
    s = case.make_session(want_norm=True)
    s.score_select(case.q_layers, case.cache_views())
    assert_status_ok()
    anchors = s.anchors.cpu().numpy()
    for l in range(w.n_layers):
        for b in range(w.n_req):
            check_anchor_band(case.raw[(l, b)], case.k[b], anchors[l, case.k_cu[b]:case.k_cu[b + 1]])
    s.build_active_sets(case.anchors_tensor())
    for l in range(w.n_layers):
        for full_prefix in (False, True):
            out, lse = run_attention(case, s, l, B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION, simt=False)
            check_attention(case, l, out, lse, full_prefix)
    # the same sizes through the persistent form: two blocks walk every item (one-tile contexts, items without work)
    s.shape.set_tuning(attention_ctx_splits=1, attention_persistent=1, attention_grid_blocks=2)
    try:
        for l in range(w.n_layers):
            for full_prefix in (False, True):
                out, lse = run_attention(case, s, l, B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION, simt=False)
                check_attention(case, l, out, lse, full_prefix)
    finally:
        s.shape.set_tuning()


def test_loose_host_bounds_give_the_same_result(case):
    """Host bounds may be loose (|R_l| <= |U| <= T_c).  With the same context split the bits are those of the
    exact bounds; when the launch size picks another split count only the summation order changes."""
    w = case.w
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    l = 0
    f = case.fresh[l]
    for forced in (1, 0):
        s.shape.set_tuning(attention_ctx_splits=forced)
        try:
            exact, _ = run_attention(case, s, l, B().CTX_UNION, simt=False)
            out = torch.zeros_like(f.q_new)
            lse = torch.zeros(w.n_q_heads, f.q_new.shape[0], dtype=torch.float32, device=case.device)
            s.attention(l, case.cache_views()[l], f.q_new, f.k_new, f.v_new, out, list(w.ctx_lens), list(w.ctx_lens), lse_out=lse)
            assert_status_ok()
        finally:
            s.shape.set_tuning()
        if forced == 1:
            assert torch.equal(out, exact)
        else:
            check_attention(case, l, out, lse, False)
            assert float((out.float() - exact.float()).abs().max()) <= 2e-2


def test_bad_index_lists_are_reported_not_faulted():
    """Out-of-range ranks are caught on the device: the status word says so, nothing faults."""
    case = Case(small_llama(n_layers=1, ctx=(512,), q=(8,)))
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    torch.cuda.synchronize()
    s.r_rank[:4] = torch.tensor([100000, -5, 100001, 100002], dtype=torch.int32, device=case.device)
    f = case.fresh[0]
    out = torch.zeros_like(f.q_new)
    s.attention(0, case.cache_views()[0], f.q_new, f.k_new, f.v_new, out, case.max_targets(0), case.max_ctx())
    st, detail = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX, (st, detail)
    st, _ = B().relaxkv_read_device_status()
    assert st == 0                                                  # reading clears the word
    k2, v2 = case.k_cache[0].clone(), case.v_cache[0].clone()
    s.scatter(0, B().CacheView(k2, v2, [0]), f.k_new, f.v_new, case.max_targets(0))
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX
    # fewer rows in q_new / out than the layer has targets (loose host bounds cannot see it): reported on the device,
    # nothing is written past the rows that exist
    s.build_active_sets(case.anchors_tensor())
    n = f.q_new.shape[0]
    short = torch.full((n - 3,) + tuple(f.q_new.shape[1:]), 3.0, dtype=f.q_new.dtype, device=case.device)
    guard = torch.full((64,) + tuple(f.q_new.shape[1:]), 5.0, dtype=f.q_new.dtype, device=case.device)
    s.attention(0, case.cache_views()[0], f.q_new[:n - 3].contiguous(), f.k_new, f.v_new, short, list(case.w.ctx_lens),
                list(case.w.ctx_lens))
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX
    assert torch.all(short == 3.0) and torch.all(guard == 5.0)


def test_expired_wait_is_reported_and_the_context_stays_usable():
    """A wait that can never be satisfied gives up after its limit: the kernel returns, the status word
    says RELAXKV_ERR_TIMEOUT, and the next call on the same context works."""
    import time
    t0 = time.time()
    B().relaxkv_debug_wait_timeout()
    st, detail = B().relaxkv_read_device_status()
    assert st == B().ERR_TIMEOUT, (st, detail)
    assert 0.2 < time.time() - t0 < 5.0
    case = Case(inputs.tiny())
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    out, lse = run_attention(case, s, 0, B().CTX_UNION, simt=False)
    check_attention(case, 0, out, lse, False)


@pytest.mark.parametrize("given_lse", [False, True], ids=["both_passes", "given_lse"])
@pytest.mark.parametrize("head_dim", [128, 64])
def test_scoring_after_an_expired_wait_adds_nothing_up(head_dim, given_lse):
    """While the status word says RELAXKV_ERR_TIMEOUT the scoring passes leave their partial sums alone (the workspace is zero, so the
    scores are sums of zeros) and give their tensor memory back: the same call works once the word has been read."""
    w = small_llama(n_layers=2, ctx=(1500, 300), q=(40, 8)) if head_dim == 128 else inputs.tiny()
    case = Case(w)
    s = case.make_session()
    lses = None
    if given_lse:               # (their values only have to be finite: what they scale is not looked at)
        lses = [torch.zeros(w.n_q_heads, int(case.q_cu[-1]), dtype=torch.float32, device=case.device) for _ in range(w.n_layers)]
    s.workspace.zero_()
    s.raw.fill_(3.0)
    B().relaxkv_debug_wait_timeout()
    s.score_select(case.q_layers, case.cache_views(), row_lse_layers=lses)
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_TIMEOUT
    assert torch.all(s.raw == 0)
    s.score_select(case.q_layers, case.cache_views())
    assert_status_ok()
    raw = s.raw.cpu().numpy().astype(np.float64)
    for l in range(w.n_layers):
        for b in range(w.n_req):
            ref = case.raw[(l, b)]
            assert np.all(np.abs(raw[l, case.ctx_cu[b]:case.ctx_cu[b + 1]] - ref) <= 1e-3 * ref + 1e-6 / w.ctx_lens[b])


# ------------------------------------------------ controlled configurations (explicit lists) ----

def _pack(lists, device):
    cu = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int32)
    flat = np.concatenate(lists).astype(np.int32) if sum(len(x) for x in lists) else np.zeros(0, np.int32)
    return torch.from_numpy(flat).to(device), torch.from_numpy(cu).to(device), cu


def _run_lists(case, s, l, ctx_lists, tgt_lists, fresh=None):
    """GPU list attention for per-request context / target position lists; returns out, lse, fresh tensors."""
    w = case.w
    ctx_pos, ctx_cu, _ = _pack(ctx_lists, case.device)
    tgt_pos, tgt_cu, tcu = _pack(tgt_lists, case.device)
    if fresh is None:
        qs, ks, vs = [], [], []
        for b in range(w.n_req):
            lo, hi = int(case.ctx_cu[b]), int(case.ctx_cu[b + 1])
            q, k, v = inputs.fresh_qkv(w, l, b, case.k_cache[l][lo:hi], case.v_cache[l][lo:hi],
                                       torch.from_numpy(np.asarray(tgt_lists[b], dtype=np.int64)))
            qs.append(q); ks.append(k); vs.append(v)
        fresh = (torch.cat(qs).contiguous(), torch.cat(ks).contiguous(), torch.cat(vs).contiguous())
    q_new, k_new, v_new = fresh
    out = torch.full_like(q_new, 3.0)
    lse = torch.zeros(w.n_q_heads, q_new.shape[0], dtype=torch.float32, device=case.device)
    B().relaxkv_list_attention(s.shape, case.cache_views()[l], q_new, k_new, v_new, ctx_pos, ctx_cu, tgt_pos, tgt_cu,
                               [len(x) for x in tgt_lists], [len(x) for x in ctx_lists], out, s.workspace, lse_out=lse)
    assert_status_ok()
    return out, lse, fresh, tcu


def test_list_attention_reduces_to_the_method(case):
    """Context = U and targets = R_l through the explicit-list call give the method's own output bits."""
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    l = case.w.n_layers - 1
    ref, _ = run_attention(case, s, l, B().CTX_UNION, simt=False)
    f = case.fresh[l]
    out, _, _, _ = _run_lists(case, s, l, [case.sets[b].u_pos for b in range(case.w.n_req)],
                              [case.sets[b].positions(l) for b in range(case.w.n_req)], fresh=(f.q_new, f.k_new, f.v_new))
    assert torch.equal(out, ref)


@pytest.mark.parametrize("persistent", [0, 1], ids=["auto", "persistent"])
@pytest.mark.parametrize("variant", ["global_targets", "layerwise_sparse", "global_sparse"])
def test_controlled_configurations_match_oracle(case, variant, persistent):
    w = case.w
    rng = np.random.default_rng(5)
    s = case.make_session()
    if persistent:                                # the persistent form of the kernel, two blocks walking all items
        s.shape.set_tuning(attention_ctx_splits=1, attention_persistent=1, attention_grid_blocks=2)
    l = 0
    ctx_lists, tgt_lists = [], []
    for b in range(w.n_req):
        T, st = w.ctx_lens[b], case.sets[b]
        n_u = len(st.u_pos)
        if variant == "global_targets":          # targets ranked over the whole context, not a subset of U
            g = orc.mean_scores(np.stack([orc.minmax(case.raw[(ll, b)]) for ll in range(w.n_layers)]))
            tgt = orc.topk(g, min(max(1, int(0.2 * T)), n_u))
            if T > 8:
                tgt = np.unique(np.concatenate([[0], tgt])) if st.u_pos[0] > 0 else tgt      # a target before all of U
            ctx = st.u_pos
        elif variant == "layerwise_sparse":      # U_l = top-|U| of this layer's score; the method's targets
            ctx = orc.topk(case.raw[(l, b)], n_u)
            tgt = st.positions(l)
        else:                                    # one shared context set from the across-layer mean score
            g = orc.mean_scores(np.stack([orc.minmax(case.raw[(ll, b)]) for ll in range(w.n_layers)]))
            ctx = orc.topk(g, n_u)
            tgt = st.positions(l)
        ctx_lists.append(np.asarray(ctx, dtype=np.int32)); tgt_lists.append(np.asarray(tgt, dtype=np.int32))
    out, lse, fresh, tcu = _run_lists(case, s, l, ctx_lists, tgt_lists)
    for b in range(w.n_req):
        lo, hi = int(tcu[b]), int(tcu[b + 1])
        if hi == lo:
            continue
        qn, kn, vn = (inputs.bf16_bits(t[lo:hi]) for t in fresh)
        ref, ref_lse = orc.list_attention(case.req_k(l, b), case.req_v(l, b), qn, kn, vn, ctx_lists[b], tgt_lists[b], case.scale)
        mx, mean = attention_errors(out[lo:hi], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (variant, b, mx, mean)
        got_lse = lse[:, lo:hi].cpu().numpy().astype(np.float64).T
        empty = np.isneginf(ref_lse)
        assert np.array_equal(np.isneginf(got_lse), empty)
        np.testing.assert_allclose(got_lse[~empty], ref_lse[~empty], atol=2e-3, rtol=1e-4)
    # cache update for the explicit target list, bit-exact
    k2, v2 = case.k_cache[l].clone(), case.v_cache[l].clone()
    tgt_pos, tgt_cu, _ = _pack(tgt_lists, case.device)
    B().relaxkv_scatter_kv_lists(s.shape, B().CacheView(k2, v2, [int(x) for x in case.ctx_cu[:-1]]), fresh[1], fresh[2],
                                 tgt_pos, tgt_cu, [len(x) for x in tgt_lists])
    assert_status_ok()
    k2_b, v2_b = inputs.bf16_bits(k2), inputs.bf16_bits(v2)
    for b in range(w.n_req):
        lo, hi = int(tcu[b]), int(tcu[b + 1])
        rk, rv = case.req_k(l, b).copy(), case.req_v(l, b).copy()
        orc.scatter(rk, rv, inputs.bf16_bits(fresh[1][lo:hi]), inputs.bf16_bits(fresh[2][lo:hi]), tgt_lists[b])
        np.testing.assert_array_equal(k2_b[case.ctx_cu[b]:case.ctx_cu[b + 1]], rk)
        np.testing.assert_array_equal(v2_b[case.ctx_cu[b]:case.ctx_cu[b + 1]], rv)


@pytest.mark.parametrize("bad", ["later", "next", "first"])
@pytest.mark.parametrize("tuning", [dict(attention_ctx_splits=1, attention_persistent=2), dict(attention_ctx_splits=1, attention_persistent=1),
                                    dict(attention_ctx_splits=2)], ids=["one_shot", "persistent", "split"])
def test_targets_before_their_context_are_zero_whatever_the_keys(tuning, bad):
    """A target that sees no context entry is a zero row with lse = -inf, also where the key tiles its query tile walks hold NaN or
    infinities: in entries past every target of the request, in the next request's rows behind them, or in the very first entry."""
    case = Case(small_llama(n_layers=1, ctx=(700, 400), q=(8, 8)))
    s = case.make_session()
    s.shape.set_tuning(**tuning)
    ctx_lists = [np.arange(100, 700, 3, dtype=np.int32), np.arange(5, 400, 2, dtype=np.int32)]       # 200 = 1.6 tiles, 198 entries
    early = [0, 17, 60, 99]
    tgt_lists = [np.array(early if bad == "first" else early + [250, 401, 652], dtype=np.int32), np.array([0, 6, 300], dtype=np.int32)]
    rows = {"later": [655, 658, 697], "next": [700 + 5, 700 + 7], "first": [100]}[bad]
    for i, r in enumerate(rows):
        case.k_cache[0][r] = float("nan") if i % 2 == 0 else float("inf")
    out, lse, fresh, tcu = _run_lists(case, s, 0, ctx_lists, tgt_lists)
    assert torch.all(out[:len(early)] == 0) and torch.all(torch.isneginf(lse[:, :len(early)]))
    if bad != "first":                  # the rows that see something: entries past their position do not count
        n = int(tcu[1])
        qn, kn, vn = (inputs.bf16_bits(t[:n]) for t in fresh)
        ref, _ = orc.list_attention(case.req_k(0, 0), case.req_v(0, 0), qn, kn, vn, ctx_lists[0], tgt_lists[0], case.scale)
        mx, mean = attention_errors(out[:n], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (mx, mean)


def test_mean_scores_and_global_topk(case):
    """g = mean over layers of the normalised scores (fixed summation order), then top-m of g."""
    w = case.w
    s = case.make_session(want_norm=True)
    s.score_select(case.q_layers, case.cache_views())
    g = torch.empty(int(case.ctx_cu[-1]), dtype=torch.float32, device=case.device)
    B().relaxkv_mean_scores(s.shape, w.n_layers, s.norm, g)
    norm = s.norm.cpu().numpy()
    ref = norm[0].astype(np.float32).copy()
    for l in range(1, w.n_layers):
        ref = ref + norm[l]
    ref = ref / np.float32(w.n_layers)
    np.testing.assert_array_equal(g.cpu().numpy(), ref)                      # same fp32 operations, same order
    m = [max(1, t // 5) for t in w.ctx_lens]
    anchors = torch.empty(1, sum(m), dtype=torch.int32, device=case.device)
    B().relaxkv_select_topk(s.shape, 1, m, g.view(1, -1), anchors)
    assert_status_ok()
    got = anchors.cpu().numpy()[0]
    off = 0
    for b in range(w.n_req):
        seg = ref[case.ctx_cu[b]:case.ctx_cu[b + 1]].astype(np.float64)
        np.testing.assert_array_equal(got[off:off + m[b]], orc.topk(seg, m[b]))
        off += m[b]


# ------------------------------------------- query prefill attention feeding the scoring ----

def test_query_prefill_lse_replaces_the_statistics_pass():
    """The query's own causal attention over [context, query] (the explicit-list call with every position
    as context and the query positions as targets, cache-only) yields each row's log-normaliser; given to
    relaxkv_score_select it skips the statistics pass and the scores are the attention weights of that
    wider softmax restricted to the context (the 'real forward pass' reading of the score)."""
    w = small_qwen(n_layers=1, ctx=(1100,), q=(40,))
    case = Case(w)
    T, Qn, H, Hkv, D = w.ctx_lens[0], w.q_lens[0], w.n_q_heads, w.n_kv_heads, w.head_dim
    g = torch.Generator(device="cpu").manual_seed(99)
    kq = torch.randn(Qn, Hkv, D, generator=g).to(torch.bfloat16).to(case.device)      # the query tokens' own K/V
    vq = torch.randn(Qn, Hkv, D, generator=g).to(torch.bfloat16).to(case.device)
    k_ext = torch.cat([case.k_cache[0], kq]).contiguous()
    v_ext = torch.cat([case.v_cache[0], vq]).contiguous()
    shape_ext = B().Shape(H, Hkv, D, [T + Qn], [Qn], case.scale)
    ws = torch.empty(B().relaxkv_workspace_bytes(shape_ext, 1) + 256, dtype=torch.uint8, device=case.device)
    ws = ws[(-ws.data_ptr()) % 256:]
    ctx_pos = torch.arange(T + Qn, dtype=torch.int32, device=case.device)
    tgt_pos = torch.arange(T, T + Qn, dtype=torch.int32, device=case.device)
    cu_ctx = torch.tensor([0, T + Qn], dtype=torch.int32, device=case.device)
    cu_tgt = torch.tensor([0, Qn], dtype=torch.int32, device=case.device)
    q = case.q_layers[0]
    out = torch.empty_like(q)
    lse = torch.empty(H, Qn, dtype=torch.float32, device=case.device)
    B().relaxkv_list_attention(shape_ext, B().CacheView(k_ext, v_ext, [0]), q, None, None, ctx_pos, cu_ctx, tgt_pos, cu_tgt,
                               [Qn], [T + Qn], out, ws, lse_out=lse)
    assert_status_ok()
    # oracle: the same causal attention, then scores with its log-normalisers
    kb, vb, qb = inputs.bf16_bits(k_ext), inputs.bf16_bits(v_ext), inputs.bf16_bits(q)
    ref_out, ref_lse = orc.list_attention(kb, vb, qb, None, None, np.arange(T + Qn), np.arange(T, T + Qn), case.scale)
    mx, mean = attention_errors(out, ref_out)
    assert mx <= MAX_ABS and mean <= MEAN_ABS
    np.testing.assert_allclose(lse.cpu().numpy().T, ref_lse, atol=2e-3, rtol=1e-4)
    ref_raw = orc.raw_scores(qb, kb[:T], case.scale, lse=ref_lse.T)
    s = case.make_session()
    s.score_select(case.q_layers, case.cache_views(), row_lse_layers=[lse])
    assert_status_ok()
    got = s.raw.cpu().numpy()[0].astype(np.float64)
    assert np.all(np.abs(got - ref_raw) <= 1e-3 * ref_raw + 1e-6 / T)
    assert got.sum() < 1.0                                   # part of each row's mass sits on the query's own keys
    check_anchor_band(ref_raw, case.k[0], s.anchors.cpu().numpy()[0])


def test_query_prefill_attention_emits_the_scores_of_its_own_pass():
    """relaxkv_query_prefill_attention: one call gives the query's causal attention over [context, query] (output and
    log-normalisers) AND the context scores with those normalisers - the score of the query's real forward pass.  Two
    requests with a gap between their cache rows; against the oracle's causal attention and its supplied-normaliser
    scores, and the anchors picked from the emitted scores against the oracle's top-k band."""
    H, Hkv, D = 16, 4, 128
    ctx, qn = (1100, 700), (40, 9)
    offs = [0, 1300]                                   # rows 1140..1299 belong to nobody
    rows = 1300 + 700 + 9
    scale = D ** -0.5
    g = torch.Generator(device="cpu").manual_seed(21)
    k_all = torch.randn(rows, Hkv, D, generator=g).to(torch.bfloat16).cuda()
    v_all = torch.randn(rows, Hkv, D, generator=g).to(torch.bfloat16).cuda()
    q = torch.randn(sum(qn), H, D, generator=g).to(torch.bfloat16).cuda()
    shape = B().Shape(H, Hkv, D, list(ctx), list(qn), scale)
    ext = B().Shape(H, Hkv, D, [c + n for c, n in zip(ctx, qn)], list(qn), scale)
    ws = torch.empty(B().relaxkv_workspace_bytes(ext, 1) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    out = torch.zeros_like(q)
    lse = torch.zeros(H, sum(qn), dtype=torch.float32, device="cuda")
    raw = torch.zeros(sum(ctx), dtype=torch.float32, device="cuda")
    B().relaxkv_query_prefill_attention(shape, B().CacheView(k_all, v_all, offs), q, out, lse, raw, ws)
    assert_status_ok()
    k_anchor = [B().relaxkv_anchor_count(t, 0.15) for t in ctx]
    anchors = torch.zeros(1, sum(k_anchor), dtype=torch.int32, device="cuda")
    B().relaxkv_select_topk(shape, 1, k_anchor, raw.view(1, -1), anchors)
    assert_status_ok()
    lo_q = lo_t = lo_k = 0
    for b in range(2):
        T, Qn = ctx[b], qn[b]
        kb = inputs.bf16_bits(k_all[offs[b]:offs[b] + T + Qn].contiguous())
        vb = inputs.bf16_bits(v_all[offs[b]:offs[b] + T + Qn].contiguous())
        qb = inputs.bf16_bits(q[lo_q:lo_q + Qn])
        ref_out, ref_lse = orc.list_attention(kb, vb, qb, None, None, np.arange(T + Qn), np.arange(T, T + Qn), scale)
        mx, mean = attention_errors(out[lo_q:lo_q + Qn], ref_out)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (b, mx, mean)
        np.testing.assert_allclose(lse[:, lo_q:lo_q + Qn].cpu().numpy().T, ref_lse, atol=2e-3, rtol=1e-4)
        ref_raw = orc.raw_scores(qb, kb[:T], scale, lse=ref_lse.T)
        got = raw[lo_t:lo_t + T].cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - ref_raw) <= 1e-3 * ref_raw + 1e-6 / T), np.abs(got / ref_raw - 1).max()
        assert got.sum() < 1.0                               # part of each row's mass sits on the query's own keys
        check_anchor_band(ref_raw, k_anchor[b], anchors[0, lo_k:lo_k + k_anchor[b]].cpu().numpy())
        lo_q, lo_t, lo_k = lo_q + Qn, lo_t + T, lo_k + k_anchor[b]
    # the attention alone (no scores asked for) gives the same output bits
    out2 = torch.zeros_like(q)
    B().relaxkv_query_prefill_attention(shape, B().CacheView(k_all, v_all, offs), q, out2, lse, None, ws)
    assert_status_ok()
    assert torch.equal(out, out2)


@pytest.mark.parametrize("head_major", [False, True])
@pytest.mark.parametrize("n_splits", [0, 1, 3])
def test_cache_attention_of_query_rows_and_a_decode_step(head_major, n_splits):
    """The pass after the repair loop: query rows (and a single decode token) attend to the cache's own causal
    prefix, read through the cache's strides without a gather.  Three requests in one call, token-major and
    head-major caches with a gap between the requests' rows, against the oracle's explicit-list attention with
    every position as context.  The gaps hold NaN / Inf bit patterns."""
    H, Hkv, D = 16, 4, 128
    lens, n_tgt = (1500, 300, 2200), (37, 1, 64)                 # the middle request is a decode step: one row
    offs = [0, 1600, 2000]                                        # rows 1500..1599 and 1900..1999 belong to nobody
    rows = 4300
    g = torch.Generator(device="cpu").manual_seed(5)
    k_all = torch.randn(rows, Hkv, D, generator=g).to(torch.bfloat16).cuda()
    v_all = torch.randn(rows, Hkv, D, generator=g).to(torch.bfloat16).cuda()
    # the rows that belong to nobody hold what an uninitialised slot may hold: NaN and infinities (plain data; the
    # last tile of every request reaches into them, and a masked key must not let them through)
    for lo_gap, hi_gap in ((1500, 1600), (1900, 2000), (4200, 4300)):
        k_all[lo_gap:hi_gap] = float("nan")
        v_all[lo_gap:hi_gap:2] = float("nan")
        v_all[lo_gap + 1:hi_gap:2] = float("inf")
    if head_major:
        k_all = k_all.permute(1, 0, 2).contiguous().permute(1, 0, 2)
        v_all = v_all.permute(1, 0, 2).contiguous().permute(1, 0, 2)
    q = torch.randn(sum(n_tgt), H, D, generator=g).to(torch.bfloat16).cuda()
    # targets: the last tokens of each request (the query suffix), ascending
    tgt = [np.arange(t - n, t, dtype=np.int32) for t, n in zip(lens, n_tgt)]
    tgt_pos = torch.from_numpy(np.concatenate(tgt)).cuda()
    tgt_cu = torch.tensor(np.concatenate([[0], np.cumsum(n_tgt)]).astype(np.int32)).cuda()
    shape = B().Shape(H, Hkv, D, list(lens), None, D ** -0.5, attention_ctx_splits=n_splits)
    ws = torch.empty(B().relaxkv_workspace_bytes(shape, 1) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    out = torch.zeros_like(q)
    lse = torch.zeros(H, q.shape[0], dtype=torch.float32, device="cuda")
    B().relaxkv_cache_attention(shape, B().CacheView(k_all, v_all, offs), q, tgt_pos, tgt_cu, list(n_tgt), out, ws, lse_out=lse)
    assert_status_ok()
    lo = 0
    for b in range(3):
        kb = inputs.bf16_bits(k_all[offs[b]:offs[b] + lens[b]].contiguous())
        vb = inputs.bf16_bits(v_all[offs[b]:offs[b] + lens[b]].contiguous())
        qb = inputs.bf16_bits(q[lo:lo + n_tgt[b]])
        ref, ref_lse = orc.list_attention(kb, vb, qb, None, None, np.arange(lens[b]), tgt[b], D ** -0.5)
        mx, mean = attention_errors(out[lo:lo + n_tgt[b]], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (b, mx, mean)
        np.testing.assert_allclose(lse[:, lo:lo + n_tgt[b]].cpu().numpy().T, ref_lse, atol=2e-3, rtol=1e-4)
        lo += n_tgt[b]
    # a position past the request's end is reported, not read
    bad = tgt_pos.clone()
    bad[0] = lens[0]
    B().relaxkv_cache_attention(shape, B().CacheView(k_all, v_all, offs), q, bad, tgt_cu, list(n_tgt), out, ws)
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX


@pytest.mark.parametrize("H,Hkv,D", [(8, 8, 64), (12, 4, 128), (40, 8, 128), (32, 2, 64)], ids=["g1_d64", "g3_d128", "g5_d128", "g16_d64"])
@pytest.mark.parametrize("n_splits,head_major", [(0, False), (1, True), (5, False)])
def test_decode_attention_one_token_per_request(H, Hkv, D, n_splits, head_major):
    """A decode step: at most one token per request attends to its cache prefix through the streaming kernel (TMA ring,
    warp-level MMA fragments, split merge).  Five requests in one call - contexts of 1, 33, 129, 1000 and 2049 tokens,
    the token's position anywhere in the request, one request without a token - with NaN / Inf in the rows between the
    requests, against the oracle's explicit-list attention; then a position past the request's end and a second token
    where the host promised one are reported, not read."""
    lens = (1, 33, 129, 1000, 2049)
    has = (1, 1, 0, 1, 1)
    pos = (0, 32, 0, 700, 2048)
    offs, rows = [], 0
    for t in lens:
        offs.append(rows); rows += t + 40                          # 40 rows that belong to nobody behind every request
    g = torch.Generator(device="cpu").manual_seed(9)
    k_all = torch.randn(rows, Hkv, D, generator=g).to(torch.bfloat16).cuda()
    v_all = torch.randn(rows, Hkv, D, generator=g).to(torch.bfloat16).cuda()
    for o, t in zip(offs, lens):
        k_all[o + t:o + t + 40] = float("nan")
        v_all[o + t:o + t + 40:2] = float("nan")
        v_all[o + t + 1:o + t + 40:2] = float("-inf")
    if head_major:
        k_all = k_all.permute(1, 0, 2).contiguous().permute(1, 0, 2)
        v_all = v_all.permute(1, 0, 2).contiguous().permute(1, 0, 2)
    n = sum(has)
    q = torch.randn(n + 1, H, D, generator=g).to(torch.bfloat16).cuda()        # one spare row that must stay untouched
    tgt_pos = torch.tensor([p for p, h in zip(pos, has) if h], dtype=torch.int32).cuda()
    tgt_cu = torch.tensor(np.concatenate([[0], np.cumsum(has)]).astype(np.int32)).cuda()
    shape = B().Shape(H, Hkv, D, list(lens), None, D ** -0.5, attention_ctx_splits=n_splits)
    ws = torch.empty(B().relaxkv_workspace_bytes(shape, 1) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    out = torch.full_like(q, 3.0)
    lse = torch.zeros(H, n + 1, dtype=torch.float32, device="cuda")
    view = B().CacheView(k_all, v_all, offs)
    B().relaxkv_cache_attention(shape, view, q, tgt_pos, tgt_cu, [1] * len(lens), out, ws, lse_out=lse)   # loose bound for request 2
    assert_status_ok()
    row = 0
    for b in range(len(lens)):
        if not has[b]:
            continue
        kb = inputs.bf16_bits(k_all[offs[b]:offs[b] + lens[b]].contiguous())
        vb = inputs.bf16_bits(v_all[offs[b]:offs[b] + lens[b]].contiguous())
        ref, ref_lse = orc.list_attention(kb, vb, inputs.bf16_bits(q[row:row + 1]), None, None, np.arange(lens[b]),
                                          np.array([pos[b]], dtype=np.int32), D ** -0.5)
        mx, mean = attention_errors(out[row:row + 1], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (b, mx, mean)
        np.testing.assert_allclose(lse[:, row:row + 1].cpu().numpy().T, ref_lse, atol=2e-3, rtol=1e-4)
        row += 1
    assert torch.all(out[n] == 3.0)
    bad = tgt_pos.clone()
    bad[1] = lens[1]                                               # one past the end of request 1
    B().relaxkv_cache_attention(shape, view, q, bad, tgt_cu, [1] * len(lens), out, ws)
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX
    two = torch.tensor([0, 1, 3, 3, 4, 5], dtype=torch.int32).cuda()            # request 1 brings two tokens
    guard = torch.full((6, H, D), 3.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_cache_attention(shape, view, torch.cat([q, q])[:6].contiguous(), torch.tensor([0, 5, 6, 1, 2], dtype=torch.int32).cuda(),
                                two, [1] * len(lens), guard, ws)
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX


@pytest.mark.parametrize("H,Hkv,D,lens", [
    (8, 8, 64, [12000] + [200 + 37 * i for i in range(23)]), (16, 8, 128, [130 * i + 1 for i in range(1, 12)] + [9001]),
    (5, 1, 128, [257, 385, 1, 128, 511, 4000]), (64, 64, 64, [1500, 40, 700])], ids=["24_one_long", "12_long_last", "few_tiles", "heads_fill_the_sms"])
def test_decode_attention_of_ragged_batches(H, Hkv, D, lens):
    """One token per request where the requests nearly fill the GPU or more: a long context is split beside short ones that are not,
    three tiles stay one block.  Against the oracle, and the same token without lists (a query of one token) bit for bit."""
    offs = np.concatenate([[0], np.cumsum(lens)[:-1]]).tolist()
    g = torch.Generator(device="cpu").manual_seed(12)
    k_all = torch.randn(sum(lens), Hkv, D, generator=g).to(torch.bfloat16).cuda()
    v_all = torch.randn(sum(lens), Hkv, D, generator=g).to(torch.bfloat16).cuda()
    nb = len(lens)
    q = torch.randn(nb, H, D, generator=g).to(torch.bfloat16).cuda()
    shape = B().Shape(H, Hkv, D, lens, [1] * nb, D ** -0.5)
    ws = torch.empty(B().relaxkv_workspace_bytes(shape, 1) + 256, dtype=torch.uint8, device="cuda")
    ws = ws[(-ws.data_ptr()) % 256:]
    out, lse = torch.full_like(q, 3.0), torch.zeros(H, nb, dtype=torch.float32, device="cuda")
    view = B().CacheView(k_all, v_all, offs)
    tgt_pos = torch.tensor([t - 1 for t in lens], dtype=torch.int32).cuda()
    B().relaxkv_cache_attention(shape, view, q, tgt_pos, torch.arange(nb + 1, dtype=torch.int32).cuda(), [1] * nb, out, ws, lse_out=lse)
    assert_status_ok()
    for b, (o, t) in enumerate(zip(offs, lens)):
        kb, vb = inputs.bf16_bits(k_all[o:o + t].contiguous()), inputs.bf16_bits(v_all[o:o + t].contiguous())
        ref, ref_lse = orc.list_attention(kb, vb, inputs.bf16_bits(q[b:b + 1]), None, None, np.arange(t), np.array([t - 1], dtype=np.int32), D ** -0.5)
        mx, mean = attention_errors(out[b:b + 1], ref)
        assert mx <= MAX_ABS and mean <= MEAN_ABS, (b, mx, mean)
        np.testing.assert_allclose(lse[:, b:b + 1].cpu().numpy().T, ref_lse, atol=2e-3, rtol=1e-4)
    if min(lens) > 1:
        own = B().Shape(H, Hkv, D, [t - 1 for t in lens], [1] * nb, D ** -0.5)
        out2, lse2 = torch.full_like(q, 3.0), torch.zeros_like(lse)
        B().relaxkv_query_prefill_attention(own, view, q, out2, lse2, None, ws)
        assert_status_ok()
        assert torch.equal(out, out2) and torch.equal(lse, lse2)


def _one_rank_group():
    """A process group of this one process on the GPU (NCCL): the all-reduce of the sharded path runs for real,
    over a single rank."""
    import socket
    import torch.distributed as dist
    sock = socket.socket()
    sock.bind(("127.0.0.1", 0))
    port = sock.getsockname()[1]
    sock.close()
    dist.init_process_group("nccl", init_method=f"tcp://127.0.0.1:{port}", rank=0, world_size=1,
                            device_id=torch.device("cuda", torch.cuda.current_device()))
    return dist


def test_head_sharded_path_on_one_gpu():
    """The KV-head-sharded layout, its two ranks run one after the other on this GPU (their kernels never wait on
    one another).  Selection: each shard's partial scores go through sharded.combine_partial_scores - the all-reduce
    (over this process alone, so the other shard's partial is added beforehand, which is what the reduction would
    deliver) and the library's scaling kernel, on a stream of its own - and must average to the unsharded scores;
    the anchors from the combined scores are those of the unsharded call.  Repair: gather, attention and the cache
    update on each shard's own heads (cache views k[:, lo:hi], H/N query heads) must equal the oracle's result for
    those heads, and the two shards' cache updates together the unsharded update, bit for bit."""
    from paper_2609_33503_b200 import sharded
    from paper_2609_33503_b200.pipeline import RepairSession
    case = Case(small_llama(n_layers=2, ctx=(1536,), q=(24,)))
    w = case.w
    full = case.make_session()
    full.score_select(case.q_layers, case.cache_views())
    world = 2
    side = torch.cuda.Stream()
    sessions, parts = [], []
    for rank in range(world):
        kv_lo, kv_hi, q_lo, q_hi = sharded.head_shard(w.n_q_heads, w.n_kv_heads, world, rank)
        s = RepairSession(q_hi - q_lo, kv_hi - kv_lo, w.head_dim, w.ctx_lens, w.q_lens, w.n_layers, case.k,
                          device=case.device, softmax_scale=case.scale)
        qs = [q[:, q_lo:q_hi].contiguous() for q in case.q_layers]
        views = [B().CacheView(k[:, kv_lo:kv_hi], v[:, kv_lo:kv_hi], [0]) for k, v in zip(case.k_cache, case.v_cache)]
        B().relaxkv_score_select(s.shape, qs, views, s.k, s.raw, None, s.workspace)       # the shard's partial scores
        sessions.append(s)
        parts.append(s.raw.clone())
    torch.cuda.synchronize()
    dist = _one_rank_group()
    try:
        for rank in range(world):
            s = sessions[rank]
            s.raw.copy_(parts[0] + parts[1])          # what the all-reduce over two ranks delivers to this rank
            torch.cuda.synchronize()
            sharded.combine_partial_scores(s, world, stream=side)
            B().relaxkv_select_topk(s.shape, s.n_layers, s.k, s.raw, s.anchors, stream=side)
        side.synchronize()
    finally:
        dist.destroy_process_group()
    assert_status_ok()
    for s in sessions:
        torch.testing.assert_close(s.raw, full.raw, rtol=2e-5, atol=1e-9)
        assert torch.equal(s.anchors, sessions[0].anchors)            # every rank selects the same anchors
        for l in range(w.n_layers):
            check_anchor_band(case.raw[(l, 0)], case.k[0], s.anchors[l].cpu().numpy())
    # ---- the repair half on each shard's heads, on the oracle's sets ----
    k_upd = [k.clone() for k in case.k_cache]
    v_upd = [v.clone() for v in case.v_cache]
    for rank in range(world):
        kv_lo, kv_hi, q_lo, q_hi = sharded.head_shard(w.n_q_heads, w.n_kv_heads, world, rank)
        s = sessions[rank]
        s.build_active_sets(case.anchors_tensor())
        n_u, n_r = s.counts()
        for l in range(w.n_layers):
            f = case.fresh[l]
            qn, kn, vn = f.q_new[:, q_lo:q_hi].contiguous(), f.k_new[:, kv_lo:kv_hi].contiguous(), f.v_new[:, kv_lo:kv_hi].contiguous()
            view = B().CacheView(case.k_cache[l][:, kv_lo:kv_hi], case.v_cache[l][:, kv_lo:kv_hi], [0])
            rows = sum(n_u) + 128
            kc = torch.empty(rows, kv_hi - kv_lo, w.head_dim, dtype=torch.bfloat16, device=case.device)
            vc = torch.empty_like(kc)
            s.gather(l, view, kn, vn, n_u, kc, vc)
            kt, vt = orc.mix_context(case.req_k(l, 0)[:, kv_lo:kv_hi].copy(), case.req_v(l, 0)[:, kv_lo:kv_hi].copy(),
                                     inputs.bf16_bits(kn), inputs.bf16_bits(vn), case.sets[0].u_pos, case.sets[0].ranks(l))
            np.testing.assert_array_equal(inputs.bf16_bits(kc[:n_u[0]]), kt)
            np.testing.assert_array_equal(inputs.bf16_bits(vc[:n_u[0]]), vt)
            out = torch.zeros_like(qn)
            s.attention(l, view, qn, kn, vn, out, n_r[l], n_u)
            assert_status_ok()
            ref, _ = orc.repair_attention(case.req_k(l, 0)[:, kv_lo:kv_hi].copy(), case.req_v(l, 0)[:, kv_lo:kv_hi].copy(),
                                          inputs.bf16_bits(qn), inputs.bf16_bits(kn), inputs.bf16_bits(vn),
                                          case.sets[0].u_pos, case.sets[0].ranks(l), case.scale)
            mx, mean = attention_errors(out, ref)
            assert mx <= MAX_ABS and mean <= MEAN_ABS, (rank, l, mx, mean)
            s.scatter(l, B().CacheView(k_upd[l][:, kv_lo:kv_hi], v_upd[l][:, kv_lo:kv_hi], [0]), kn, vn, n_r[l])
    assert_status_ok()
    whole = case.make_session()
    whole.build_active_sets(case.anchors_tensor())
    _, n_r = whole.counts()
    for l in range(w.n_layers):
        k2, v2 = case.k_cache[l].clone(), case.v_cache[l].clone()
        whole.scatter(l, B().CacheView(k2, v2, [0]), case.fresh[l].k_new, case.fresh[l].v_new, n_r[l])
        assert torch.equal(k2, k_upd[l]) and torch.equal(v2, v_upd[l])


def test_one_chunk_reading_fresh_states_equal_to_the_cache():
    """With a single chunk nothing precedes the chunk, so recomputing a token gives back its cached K/V.  Then
    (i) the cache update leaves the cache bit-identical, (ii) attention over the mixed fresh/cached context equals
    attention over the cache alone bit for bit, and (iii) at an anchor ratio of 100 % the output is dense causal
    attention over the cache, i.e. a plain prefix prefill (checked against causal attention in float64)."""
    for ratio in (0.3, 1.0):
        w = small_qwen(n_layers=2, ctx=(900,), q=(16,)).replace(ratio=ratio)
        case = Case(w)
        s = case.make_session()
        s.build_active_sets(case.anchors_tensor())
        n_u, n_r = s.counts()
        for l in range(w.n_layers):
            pos = torch.from_numpy(case.sets[0].positions(l).astype(np.int64)).to(case.device)
            f = case.fresh[l]
            k_same, v_same = case.k_cache[l][pos].contiguous(), case.v_cache[l][pos].contiguous()
            view = case.cache_views()[l]
            mixed = torch.zeros_like(f.q_new)
            s.attention(l, view, f.q_new, k_same, v_same, mixed, n_r[l], n_u)
            alone = torch.zeros_like(f.q_new)
            s.attention(l, view, f.q_new, None, None, alone, n_r[l], n_u)
            assert_status_ok()
            assert torch.equal(mixed, alone)
            k2, v2 = case.k_cache[l].clone(), case.v_cache[l].clone()
            s.scatter(l, B().CacheView(k2, v2, [0]), k_same, v_same, n_r[l])
            assert torch.equal(k2, case.k_cache[l]) and torch.equal(v2, case.v_cache[l])
            if ratio == 1.0:
                assert n_r[l] == [900] and n_u == [900]
                G = w.group
                q64 = f.q_new.double().cpu().permute(1, 0, 2).unsqueeze(0)
                k64 = case.k_cache[l].double().cpu().repeat_interleave(G, dim=1).permute(1, 0, 2).unsqueeze(0)
                v64 = case.v_cache[l].double().cpu().repeat_interleave(G, dim=1).permute(1, 0, 2).unsqueeze(0)
                ref = torch.nn.functional.scaled_dot_product_attention(q64, k64, v64, is_causal=True, scale=case.scale)[0].permute(1, 0, 2)
                d = (mixed.double().cpu() - ref).abs()
                assert d.max().item() <= MAX_ABS and d.mean().item() <= MEAN_ABS


def test_list_call_with_more_context_than_its_host_bound_is_reported():
    """Explicit lists whose true context count exceeds the host bound: the rows past the bound have no entry in the
    fresh-row map, so the gather must not use one (it zero-fills them) and the status word reports the overflow."""
    case = Case(small_llama(n_layers=1, ctx=(512,), q=(8,)))
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    sets = case.sets[0]
    ctx_list, tgt_list = sets.u_pos.astype(np.int32), sets.positions(0).astype(np.int32)
    f = case.fresh[0]
    ctx_pos, ctx_cu, _ = _pack([ctx_list], case.device)
    tgt_pos, tgt_cu, _ = _pack([tgt_list], case.device)
    s.workspace.view(torch.int32).fill_(0x7fffff00)            # stale words a trusting kernel would index with
    out = torch.zeros_like(f.q_new)
    B().relaxkv_list_attention(s.shape, case.cache_views()[0], f.q_new, f.k_new, f.v_new, ctx_pos, ctx_cu, tgt_pos, tgt_cu,
                               [len(tgt_list)], [len(ctx_list) - 40], out, s.workspace)
    st, detail = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX, (st, detail)
    out2 = torch.zeros_like(f.q_new)                           # the context stays usable: the same call with a true bound
    B().relaxkv_list_attention(s.shape, case.cache_views()[0], f.q_new, f.k_new, f.v_new, ctx_pos, ctx_cu, tgt_pos, tgt_cu,
                               [len(tgt_list)], [len(ctx_list)], out2, s.workspace)
    assert_status_ok()
    ref, _ = case.oracle_attention(0, 0)
    mx, mean = attention_errors(out2, ref)
    assert mx <= MAX_ABS and mean <= MEAN_ABS


# ------------------------------------------------ other head geometries and cache layouts ----

@pytest.mark.parametrize("H,Hkv,D,head_major", [(8, 8, 128, False), (16, 8, 64, True), (16, 2, 128, False),
                                                (32, 2, 64, False), (12, 4, 128, True)])
def test_other_geometries_and_head_major_cache(H, Hkv, D, head_major):
    """Group sizes 1, 2, 8, 16 and 3 (the last does not divide 128), both head dims, and a cache stored
    [H_kv, tokens, D] (read through its strides by the TMA-based scoring kernel and by the gather)."""
    base = inputs.Workload("geom", 2, H, Hkv, D, 64, (700, 333), (21, 9), 0.2, base_seed=7,
                           planted_chunks=((1, 6), (2,)), variant="calibrated")
    case = Case(base, head_major_cache=head_major)
    w = case.w
    s = case.make_session(want_norm=True)
    s.score_select(case.q_layers, case.cache_views())
    assert_status_ok()
    raw = s.raw.cpu().numpy().astype(np.float64)
    anchors = s.anchors.cpu().numpy()
    for l in range(w.n_layers):
        for b in range(w.n_req):
            ref = case.raw[(l, b)]
            got = raw[l, case.ctx_cu[b]:case.ctx_cu[b + 1]]
            assert np.all(np.abs(got - ref) <= 1e-3 * ref + 1e-6 / w.ctx_lens[b]), np.abs(got / ref - 1).max()
            check_anchor_band(ref, case.k[b], anchors[l, case.k_cu[b]:case.k_cu[b + 1]])
    s.build_active_sets(case.anchors_tensor())
    for l in range(w.n_layers):
        for full_prefix in (False, True):
            out, lse = run_attention(case, s, l, B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION, simt=False)
            check_attention(case, l, out, lse, full_prefix)


@pytest.mark.parametrize("G,D", [(1, 64), (3, 128), (5, 128), (7, 64), (11, 128), (16, 64)])
def test_targets_at_the_edges_of_a_pair_of_query_tiles(G, D):
    """A pair of query tiles is 256 rows of floor(256 / G) whole targets; where 128 is no multiple of G one target has heads in both
    tiles.  Target counts around one tile, one pair and two, all three forms of the launch."""
    pair = 256 // G
    for n in sorted({1, 128 // G, 128 // G + 1, pair - 1, pair, pair + 1, 2 * pair, 2 * pair + 1}):
        w = inputs.Workload("pairs", 1, 2 * G, 2, D, 64, (600,), (4,), 0.1, base_seed=n)
        pos = np.sort(np.random.default_rng(n).choice(600, n, replace=False)).astype(np.int32)
        case = Case(w, anchors_override=[[pos]])
        case.k = [n]
        s = case.make_session()
        s.build_active_sets(case.anchors_tensor())
        outs = []
        for tuning in (dict(attention_ctx_splits=1, attention_persistent=2), dict(attention_ctx_splits=1, attention_persistent=1),
                       dict(attention_ctx_splits=3)):
            s.shape.set_tuning(**tuning)
            for full_prefix in (False, True):
                out, lse = run_attention(case, s, 0, B().CTX_FULL_PREFIX if full_prefix else B().CTX_UNION, simt=False)
                check_attention(case, 0, out, lse, full_prefix)
                outs.append(out)
        assert torch.equal(outs[0], outs[2]) and torch.equal(outs[1], outs[3])


@pytest.mark.parametrize("H,Hkv,D,ctx,targets", [(4, 1, 64, (4000,), 4000), (4, 1, 64, (2600, 130, 3100), 3100), (5, 1, 128, (4500,), 4500),
                                                 (8, 2, 128, (6000,), 1229), (6, 2, 64, (5000, 3000), 400)],
                         ids=["one", "ragged", "five_heads", "few_targets", "few_targets_ragged"])
def test_longest_pairs_in_pieces(H, Hkv, D, ctx, targets):
    """A call of few tile pairs cuts its longest ones into pieces and merges them: against the oracle, with exact and with loose host
    bounds, beside the whole form (other bits: pieces were taken), and refused where a count is above its bound."""
    w = inputs.Workload("pieces", 1, H, Hkv, D, 64, ctx, (4,) * len(ctx), 0.1, base_seed=H)
    case = Case(w, anchors_override=[[np.arange(1, dtype=np.int32) for _ in ctx]])
    rng = np.random.default_rng(len(ctx))
    tgt = [np.sort(rng.choice(t, min(t, targets), replace=False)).astype(np.int32) for t in ctx]
    ctx_lists = [np.unique(np.concatenate([x, rng.choice(t, (5 * t) // 6, replace=False)])).astype(np.int32) for x, t in zip(tgt, ctx)]
    ctx_pos, ctx_cu, _ = _pack(ctx_lists, case.device)
    tgt_pos, tgt_cu, tcu = _pack(tgt, case.device)
    fresh = [torch.cat(x).contiguous() for x in zip(*[inputs.fresh_qkv(w, 0, b, case.k_cache[0][case.ctx_cu[b]:case.ctx_cu[b + 1]],
                                                                      case.v_cache[0][case.ctx_cu[b]:case.ctx_cu[b + 1]],
                                                                      torch.from_numpy(tgt[b].astype(np.int64))) for b in range(len(ctx))])]
    refs = [orc.list_attention(case.req_k(0, b), case.req_v(0, b), *(inputs.bf16_bits(t[tcu[b]:tcu[b + 1]]) for t in fresh), ctx_lists[b], tgt[b],
                               case.scale) for b in range(len(ctx))]
    n_t, n_c = [len(x) for x in tgt], [len(x) for x in ctx_lists]
    outs = []
    for tuning, max_t, max_c in ((dict(), n_t, n_c), (dict(), ctx, ctx), (dict(attention_ctx_splits=1), n_t, n_c), (dict(), [max(1, n - 1) for n in n_t], n_c)):
        shape = B().Shape(H, Hkv, D, ctx, None, case.scale, **tuning)
        ws = torch.empty(B().relaxkv_workspace_bytes(shape, 1), dtype=torch.uint8, device="cuda")
        out, lse = torch.full_like(fresh[0], 3.0), torch.zeros(H, fresh[0].shape[0], dtype=torch.float32, device="cuda")
        B().relaxkv_list_attention(shape, case.cache_views()[0], *fresh, ctx_pos, ctx_cu, tgt_pos, tgt_cu, max_t, max_c, out, ws, lse_out=lse)
        outs.append(out)
        if len(outs) == 4:
            break
        assert_status_ok()
        for b, (ref, ref_lse) in enumerate(refs):
            lo, hi = int(tcu[b]), int(tcu[b + 1])
            mx, mean = attention_errors(out[lo:hi], ref)
            assert mx <= MAX_ABS and mean <= MEAN_ABS, (b, mx, mean)
            np.testing.assert_allclose(lse[:, lo:hi].cpu().numpy().astype(np.float64).T, ref_lse, atol=2e-3, rtol=1e-4)
    assert not torch.equal(outs[0], outs[2])
    assert B().relaxkv_read_device_status()[0] == B().ERR_BAD_INDEX
    refused = torch.cat([torch.full((n,), n > 1) for n in n_t]).cuda()
    assert torch.all(outs[3][refused] == 3.0)


@pytest.mark.parametrize("n,H,Hkv,D", [(1, 8, 2, 128), (51, 40, 8, 128), (127, 8, 2, 128), (128, 32, 8, 128), (129, 8, 2, 64), (300, 40, 8, 128),
                                       (2458, 32, 8, 128), (2500, 8, 8, 64)])
def test_a_context_of_fresh_rows_alone_is_read_in_place(n, H, Hkv, D):
    """One request whose layer renews its whole context (exact bounds): the fresh rows are the context.  The same bits as by the general way
    (a bound that is one too large), whatever lies behind the rows and in the workspace, and nothing but the lists decides: equal bounds
    over a layer that renews less take the general way."""
    from paper_2609_33503_b200.pipeline import RepairSession
    b, T = B(), n + 1700
    gen = torch.Generator(device="cuda").manual_seed(n)
    normal = lambda *s: torch.randn(*s, device="cuda", generator=gen).to(torch.bfloat16)
    few = max(1, n - 3)
    s = RepairSession(H, Hkv, D, [T], [4], 2, [n])
    pos = torch.randperm(T, device="cuda", generator=gen)[:n].sort().values.to(torch.int32)
    # layer 0 renews all n, layer 1 the first `few` of them
    s.u_pos[:n] = pos
    s.u_cu.copy_(torch.tensor([0, n], dtype=torch.int32))
    ranks = torch.cat([torch.arange(n), torch.arange(n - few, n)]).to(torch.int32).cuda()
    s.r_rank[:n + few] = ranks
    s.r_cu.copy_(torch.tensor([0, n, n + few], dtype=torch.int32))
    cache = b.CacheView(normal(T, Hkv, D), normal(T, Hkv, D), [0])

    def rows(m, heads):                                      # with NaN behind them
        t = torch.full((m + 200, heads, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        t[:m] = normal(m, heads, D)
        return t[:m]
    q, k, v = rows(n, H), rows(n, Hkv), rows(n, Hkv)

    def run(layer, n_r, bound_r, bound_u):
        s.workspace.fill_(0xFF)
        out, lse = torch.zeros(n_r, H, D, dtype=torch.bfloat16, device="cuda"), torch.zeros(H, n_r, device="cuda")
        s.attention(layer, cache, q[:n_r], k[:n_r], v[:n_r], out, [bound_r], [bound_u], lse_out=lse)
        assert_status_ok()
        return out, lse
    got, want = run(0, n, n, n), run(0, n, n, n + 1)
    assert torch.isfinite(got[0]).all() and torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    if H == Hkv:                                             # an output in the place of the fresh values
        v_kept = v.clone()
        s.attention(0, cache, q, k, v, v, [n], [n])
        assert_status_ok()
        assert torch.equal(v, want[0])
        v.copy_(v_kept)
    if few < n:
        want = run(1, few, few, n)
        got = run(1, n, n, n)                                # rows past the layer's own stay as they were
        assert torch.isfinite(got[0]).all() and torch.equal(got[0][:few], want[0]) and not got[0][few:].any()
        lists = s.r_rank.clone()
        s.r_rank[1] = 0                                      # a rank twice: no list of the schedule
        s.attention(0, cache, q, k, v, torch.empty(n, H, D, dtype=torch.bfloat16, device="cuda"), [n], [n])
        status, detail = b.relaxkv_read_device_status()
        assert status == b.ERR_BAD_INDEX
        s.r_rank.copy_(lists)


def _merged_calls(form):
    """A call whose context is split over blocks and merged: H, the rows per request, run(out, lse, bounds) and the call's own bounds.  form:
    "pieces" (the longest pairs alone), "splits" (every pair, in three), each "_lists" or "_sets"; "query" (a query's rows over six key
    tiles, no lists); "decode" (a token per request); "cache" (rows at given positions of the cache)."""
    b, g = B(), torch.Generator(device="cuda").manual_seed(len(form))
    normal = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    i32 = lambda x: torch.tensor(np.asarray(x, dtype=np.int32)).cuda()
    if form in ("query", "decode", "cache"):
        H, Hkv, D, ctx, n = {"query": (8, 2, 128, (700, 640), (30, 9)), "decode": (8, 2, 64, (900, 2000, 700), (1, 1, 1)),
                             "cache": (8, 4, 128, (500, 130, 900), (40, 1, 70))}[form]
        room = [c + m for c, m in zip(ctx, n)]
        shape = b.Shape(H, Hkv, D, list(ctx) if form == "query" else room, list(n), attention_ctx_splits=0 if form == "query" else 4)
        ext = b.Shape(H, Hkv, D, room, list(n))
        view = b.CacheView(normal(sum(room), Hkv, D), normal(sum(room), Hkv, D), [sum(room[:i]) for i in range(len(n))])
        q = normal(sum(n), H, D)
        ws = torch.zeros(max(b.relaxkv_workspace_bytes(s, 1) for s in (shape, ext)), dtype=torch.uint8, device="cuda")
        tgt_cu = i32(np.concatenate([[0], np.cumsum(n)]))

        def run(out, lse, pos, counts=n):
            ws.zero_()
            rows = out.shape[0]
            if form == "query":
                b.relaxkv_query_prefill_attention(shape, view, q, out, lse, None, ws)
            else:
                b.relaxkv_cache_attention(shape, view, q[:rows], i32(pos), tgt_cu, counts, out, ws, lse_out=lse)
        if form == "cache":
            return H, D, n, lambda out, lse, counts: run(out, lse, np.concatenate([c + np.arange(m) for c, m in zip(ctx, n)]), counts), (list(n),)
        return H, D, n, run, (list(ctx),)
    H, Hkv, D, ctx = 4, 1, 64, (2600, 130, 3100) if form.startswith("pieces") else (300, 130, 250)
    cu = i32(np.concatenate([[0], np.cumsum(ctx)]))
    pos = i32(np.concatenate([np.arange(t) for t in ctx]))                   # every position is an entry and a target
    shape = b.Shape(H, Hkv, D, list(ctx), None, attention_ctx_splits=3 if form.startswith("splits") else 0)
    view = b.CacheView(normal(sum(ctx), Hkv, D), normal(sum(ctx), Hkv, D), [sum(ctx[:i]) for i in range(3)])
    q, k, v = normal(sum(ctx), H, D), normal(sum(ctx), Hkv, D), normal(sum(ctx), Hkv, D)
    ws = torch.zeros(b.relaxkv_workspace_bytes(shape, 1), dtype=torch.uint8, device="cuda")

    def run(out, lse, max_t, max_c):
        ws.zero_()
        rows = out.shape[0]
        if form.endswith("lists"):
            b.relaxkv_list_attention(shape, view, q[:rows], k, v, pos, cu, pos, cu, max_t, max_c, out, ws, lse_out=lse)
        else:
            b.relaxkv_sparse_ctx_attention(shape, b.CTX_UNION, view, q[:rows], k, v, pos, cu, pos, cu, max_t, max_c, out, ws, lse_out=lse)
    return H, D, ctx, run, (list(ctx), list(ctx))


_MERGED = ["pieces_lists", "pieces_sets", "splits_lists", "splits_sets", "cache", "decode"]


def _filled(n, H, D):
    return torch.full((n, H, D), 3.0, dtype=torch.bfloat16, device="cuda"), torch.full((H, n), 3.0, dtype=torch.float32, device="cuda")


@pytest.mark.parametrize("form,what", [(f, w) for f in _MERGED[:4] for w in ("targets", "context", "rows")] +
                         [("cache", "targets"), ("cache", "rows"), ("decode", "rows"), ("decode", "position")])
def test_a_refused_request_of_a_merged_call_keeps_its_rows(form, what):
    """The last request's targets or context entries are above their host bound, its rows past the output's end, or its token's position
    past the cache: reported, its rows of out and lse untouched (the workspace holds zeros, whose merge would be a zero row), the
    other requests' rows as in the call without the fault."""
    H, D, n, run, bounds = _merged_calls(form)
    want = _filled(sum(n), H, D)
    run(*want, *bounds)
    assert_status_ok()
    rows = sum(n) - ((5 if n[-1] > 5 else 1) if what == "rows" else 0)
    got = _filled(rows, H, D)
    wrong = [list(x) for x in bounds]
    if what != "rows":
        wrong[1 if what == "context" else 0][-1] += {"position": 1}.get(what, -1)
    run(*got, *wrong)
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX
    lo = sum(n[:-1])
    assert torch.equal(got[0][:lo], want[0][:lo]) and torch.equal(got[1][:, :lo], want[1][:, :lo])
    assert torch.all(got[0][lo:] == 3.0) and torch.all(got[1][:, lo:] == 3.0)


@pytest.mark.parametrize("form", _MERGED + ["query"])
def test_a_merged_call_after_an_expired_wait_writes_nothing(form):
    """While the status word says RELAXKV_ERR_TIMEOUT the blocks leave no partial results, and nothing is merged; once the word has
    been read the same call has its results."""
    H, D, n, run, bounds = _merged_calls(form)
    want, got = _filled(sum(n), H, D), _filled(sum(n), H, D)
    run(*want, *bounds)
    assert_status_ok()
    assert not torch.any(want[1] == 3.0)
    B().relaxkv_debug_wait_timeout()
    run(*got, *bounds)
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_TIMEOUT
    assert torch.all(got[0] == 3.0) and torch.all(got[1] == 3.0)
    run(*got, *bounds)
    assert_status_ok()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_the_forms_of_a_call_that_is_cut_have_the_same_bits():
    """A call of more tile pairs than SMs whose longest are cut: attention_persistent = 0, 1 and 2 give the same bits, which are not the whole
    form's; a number of blocks of the persistent form is one of a call that is not cut, and gives the bits of the whole form."""
    b, T = B(), 12000
    g = torch.Generator(device="cuda").manual_seed(3)
    normal = lambda: torch.randn(T, 4, 64, device="cuda", generator=g).to(torch.bfloat16)
    view, q, k, v = b.CacheView(normal(), normal(), [0]), normal(), normal(), normal()
    pos, cu = torch.arange(T, dtype=torch.int32, device="cuda"), torch.tensor([0, T], dtype=torch.int32, device="cuda")

    def run(**tuning):
        shape = b.Shape(4, 4, 64, [T], None, **tuning)
        ws = torch.empty(b.relaxkv_workspace_bytes(shape, 1), dtype=torch.uint8, device="cuda")
        out, lse = torch.empty_like(q), torch.empty(4, T, device="cuda")
        b.relaxkv_list_attention(shape, view, q, k, v, pos, cu, pos, cu, [T], [T], out, ws, lse_out=lse)
        assert_status_ok()
        return out, lse
    same = lambda x, y: torch.equal(x[0], y[0]) and torch.equal(x[1], y[1])
    cut, whole = run(), run(attention_ctx_splits=1)
    assert not same(cut, whole) and (cut[0].float() - whole[0].float()).abs().max() <= MAX_ABS
    for persistent in (1, 2):
        assert same(run(attention_persistent=persistent), cut)
        assert same(run(attention_persistent=persistent, attention_ctx_splits=1), whole)
    for blocks in (3, 100):
        assert same(run(attention_grid_blocks=blocks), whole)


@pytest.mark.parametrize("H,Hkv,D,T,n", [(8, 2, 128, 700, 300), (10, 2, 64, 500, 333), (8, 8, 64, 300, 1)])
@pytest.mark.parametrize("tuning", [dict(attention_ctx_splits=1, attention_persistent=2), dict(attention_ctx_splits=1, attention_persistent=1), dict(attention_ctx_splits=3)],
                         ids=["one_shot", "persistent", "split"])
def test_an_output_that_is_not_32_byte_aligned(H, Hkv, D, T, n, tuning):
    """Outputs are stored as whole 32-byte sectors where the output begins on one and in 16-byte pieces elsewhere: the same bits, and nothing
    written beside the rows."""
    b, g = B(), torch.Generator(device="cuda").manual_seed(n)
    normal = lambda *s: torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16)
    i32 = lambda x: torch.tensor(np.asarray(x, dtype=np.int32)).cuda()
    shape = b.Shape(H, Hkv, D, [T], None, **tuning)
    view, q, k, v = b.CacheView(normal(T, Hkv, D), normal(T, Hkv, D), [0]), normal(n, H, D), normal(n, Hkv, D), normal(n, Hkv, D)
    ws = torch.empty(b.relaxkv_workspace_bytes(shape, 1), dtype=torch.uint8, device="cuda")
    pos, tgt = i32(np.arange(T)), np.sort(np.random.default_rng(n).choice(T, n, replace=False))
    got = []
    for off in (0, 8, 16, 24):                                       # elements of two bytes
        buf = torch.full((n * H * D + 48,), 3.0, dtype=torch.bfloat16, device="cuda")
        assert buf.data_ptr() % 32 == 0
        out = buf[16 + off:16 + off + n * H * D].view(n, H, D)
        b.relaxkv_sparse_ctx_attention(shape, b.CTX_UNION, view, q, k, v, pos, i32([0, T]), i32(tgt), i32([0, n]), [n], [T], out, ws)
        assert_status_ok()
        assert torch.all(buf[:16 + off] == 3.0) and torch.all(buf[16 + off + n * H * D:] == 3.0)
        got.append(out.clone())
    assert all(torch.equal(x, got[0]) for x in got[1:])
    assert not torch.any((got[0] == 3.0).all(dim=2))
