"""GPU parity of the dense block work of the active targets (Algorithm 1, steps 14/16/20) against the fp64
block oracle, operation by operation on identical bf16 inputs, then one whole layer of the repair loop.

Tolerances: every kernel rounds its output to bf16 once (relative 2^-9) after fp32 arithmetic, so
|gpu - ref| <= 2^-8 * |ref| + abs_floor, with abs_floor scaled to the magnitude of the sum being rounded."""
import numpy as np
import pytest
import torch

from oracle import relaxkv_block_oracle as blk
from oracle import relaxkv_oracle as orc
from paper_2609_33503_b200 import inputs

pytestmark = pytest.mark.gpu


def B():
    from paper_2609_33503_b200 import binding
    return binding


def bits(t):
    return inputs.bf16_bits(t)


def rnd(*shape, scale=1.0, seed=0):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return (torch.randn(*shape, generator=g) * scale).to(torch.bfloat16).cuda()


def close(got: torch.Tensor, ref: np.ndarray, abs_floor: float):
    g = got.float().cpu().numpy().astype(np.float64)
    err = np.abs(g - ref)
    assert np.all(err <= 2.0 ** -8 * np.abs(ref) + abs_floor), float((err - 2.0 ** -8 * np.abs(ref)).max())


@pytest.mark.parametrize("M,N,K,res", [(300, 512, 320, False), (129, 264, 72, True), (1000, 1024, 2048, True), (1, 8, 8, False),
                                       (257, 1280, 640, False), (5000, 2304, 1024, True), (2, 520, 1032, True), (4, 136, 264, False)])
def test_linear(M, N, K, res):
    """Both GEMM kernels: SM pairs (256 x 256 tiles per cluster; here 129, 1000 and 5000 rows) and the single-block
    one the library picks when an odd, small number of 128-row tiles would leave half a cluster idle (300, 257, 1)."""
    _check_linear(M, N, K, res)


def _check_linear(M, N, K, res):
    x, w = rnd(M, K, seed=1), rnd(N, K, scale=K ** -0.5, seed=2)
    r = rnd(M, N, seed=3) if res else None
    y = torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear(x, w, y, residual=r)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    ref = blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), blk.f64(bits(r)) if res else None)
    close(y, ref, abs_floor=2e-3)
    torch.testing.assert_close(y.float(), (x.float() @ w.float().T + (r.float() if res else 0)), rtol=2e-2, atol=2e-2)


@pytest.mark.parametrize("M", [1, 3, 5, 64, 128, 300, 1000])
@pytest.mark.parametrize("n_q,n_kv,K", [(512, 128, 512), (5120, 1024, 5120), (320, 72, 264), (352, 96, 520)])
def test_linear_qkv_writes_the_three_projections(M, n_q, n_kv, K):
    """The fused Q/K/V projection (stacked weight, three output buffers) through its three routes - the streaming
    kernel (one row, three with a K below 4096), the cluster split-K kernel (up to 128 rows: segment boundaries inside a tile at the odd
    shape), one large GEMM whose epilogue writes the three buffers (300 rows: the single-block kernel, 1000 rows: SM pairs; widths
    that are multiples of 32, also with boundaries inside a 256-column tile) or three large GEMMs (other widths) -
    against the oracle's linear per projection; bytes around the outputs stay untouched."""
    x = rnd(M, K, seed=11)
    wq, wk, wv = rnd(n_q, K, scale=K ** -0.5, seed=12), rnd(n_kv, K, scale=K ** -0.5, seed=13), rnd(n_kv, K, scale=K ** -0.5, seed=14)
    w_qkv = B().stack_qkv(wq, wk, wv)
    bufs = [torch.full((M + 2, n), 7.0, dtype=torch.bfloat16, device="cuda") for n in (n_q, n_kv, n_kv)]
    q, k, v = (b[1:M + 1] for b in bufs)
    B().relaxkv_linear_qkv(x, w_qkv, q, k, v)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    for out, w, buf in ((q, wq, bufs[0]), (k, wk, bufs[1]), (v, wv, bufs[2])):
        ref = blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None)
        close(out, ref, abs_floor=2e-3)
        assert torch.all(buf[0] == 7.0) and torch.all(buf[M + 1] == 7.0)
        if M <= 4:                                   # the order of the sums goes by K alone: the bits of the single projection
            one = torch.empty_like(out)
            B().relaxkv_linear(x, w, one)
            assert torch.equal(one, out)


@pytest.mark.parametrize("M,N,K,res", [(5, 8, 8, False), (17, 136, 72, True), (100, 1000, 520, True), (128, 5120, 1032, False),
                                       (64, 264, 5120, True), (128, 19200, 64, False), (33, 2048, 17408, True)])
def test_linear_of_a_few_rows(M, N, K, res):
    """5 to 128 rows: tiles of 128 weight rows whose K range is split over a thread-block cluster (1 to 8 blocks, by the
    number of tiles and K blocks) and summed through distributed shared memory; ragged N and K tails, a residual
    that aliases the output, K shorter than two blocks per cluster member, more tiles than SMs (19200 / 128 =
    150: one block each, two per SM); run twice: bit-identical (the partial sums are added in rank order)."""
    x, w = rnd(M, K, seed=41), rnd(N, K, scale=K ** -0.5, seed=42)
    r = rnd(M, N, seed=43) if res else None
    y = r.clone() if res else torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear(x, w, y, residual=y if res else None)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    ref = blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), blk.f64(bits(r)) if res else None)
    close(y, ref, abs_floor=4e-3)
    y2 = r.clone() if res else torch.empty_like(y)
    B().relaxkv_linear(x, w, y2, residual=y2 if res else None)
    assert torch.equal(y, y2)


@pytest.mark.parametrize("M,N,K,swiglu", [
    (2, 264, 8200, False), (3, 1000, 4104, False), (4, 19208, 4096, False), (16, 136, 72, False), (64, 5128, 1032, False),
    (65, 5128, 1032, False), (128, 37896, 136, False), (2, 256, 4104, True), (3, 512, 2056, True), (5, 256, 72, True),
    (17, 1280, 520, True), (64, 512, 264, True), (65, 38144, 136, True), (128, 2048, 1032, True)])
def test_weight_tiles_against_a_few_rows(M, N, K, swiglu):
    """The 128-weight-row tiles at the edges of their choices: rows that fill and just pass an MMA width (16, 64), the two- and
    the one-block form (64 / 65 rows), more tiles than blocks fit (150 and 297), one to eight blocks per tile (K from 72 to
    8200), ragged last tiles and K blocks, and gate/up pairs; rows around the output stay untouched.  The fp32 sums of K
    products of N(0,1) x N(0,1/K) err by less than 2e-3 absolute at these K in any order, a bf16 rounding on top."""
    x, w = rnd(M, K, seed=51), rnd(N, K, scale=K ** -0.5, seed=52)
    buf = torch.full((M + 2, N // 2 if swiglu else N), 7.0, dtype=torch.bfloat16, device="cuda")
    y = buf[1:M + 1]
    if swiglu:
        B().relaxkv_linear_swiglu(x, B().tile_gate_up(w), y)
        ref = blk.swiglu(blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None))
    else:
        B().relaxkv_linear(x, w, y)
        ref = blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    close(y, ref, abs_floor=2e-3)
    assert torch.all(buf[0] == 7.0) and torch.all(buf[M + 1] == 7.0)


@pytest.mark.parametrize("M", [2, 3, 4])
@pytest.mark.parametrize("n_q,n_kv,K", [(8192, 1024, 5120), (8192, 1024, 8192), (5120, 1024, 4104), (1024, 128, 4096), (20480, 4096, 8200), (2048, 264, 2056)])
def test_stacked_projections_give_the_bits_of_single_ones(M, n_q, n_kv, K):
    """Two to four rows: the stacked matrix has more tiles than its parts and is shared by other numbers of blocks (8, 4, 2 and 1 for
    these), the sums over K have the same order: equal bits, and both against the oracle."""
    x = rnd(M, K, seed=61)
    ws = [rnd(n, K, scale=K ** -0.5, seed=62 + i) for i, n in enumerate((n_q, n_kv, n_kv))]
    outs = [torch.full((M, n), 7.0, dtype=torch.bfloat16, device="cuda") for n in (n_q, n_kv, n_kv)]
    B().relaxkv_linear_qkv(x, B().stack_qkv(*ws), *outs)
    for w, out in zip(ws, outs):
        one = torch.full_like(out, 7.0)
        B().relaxkv_linear(x, w, one)
        assert torch.equal(one, out)
        close(out[:, -200:], blk.linear(blk.f64(bits(x)), blk.f64(bits(w[-200:].contiguous())), None), abs_floor=2e-3)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)


@pytest.mark.parametrize("n_q,n_kv,K", [(264, 8, 3576), (2368, 8, 3584), (264, 136, 4088), (4096, 512, 4096), (264, 8, 4104), (264, 8, 8184), (1024, 264, 8192),
                                        (2400, 264, 16376), (1024, 264, 16384)])
def test_one_row_by_the_features_of_a_warp(n_q, n_kv, K):
    """One row: a stacked matrix and its pieces, on both sides of K = 3584, 4096, 8192 and 16384: equal bits, rows around the output
    untouched, and against the oracle."""
    x = rnd(1, K, seed=71)
    ws = [rnd(n, K, scale=K ** -0.5, seed=72 + i) for i, n in enumerate((n_q, n_kv, n_kv))]
    outs = [torch.full((1, n), 7.0, dtype=torch.bfloat16, device="cuda") for n in (n_q, n_kv, n_kv)]
    B().relaxkv_linear_qkv(x, B().stack_qkv(*ws), *outs)
    for w, out in zip(ws, outs):
        one, res = torch.full((3, w.shape[0]), 7.0, dtype=torch.bfloat16, device="cuda"), rnd(1, w.shape[0], seed=75)
        B().relaxkv_linear(x, w, one[1:2])
        assert torch.equal(one[1:2], out) and (one[0] == 7.0).all() and (one[2] == 7.0).all()
        ref = blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None)
        close(out, ref, abs_floor=2e-3)
        B().relaxkv_linear(x, w, one[1:2], residual=res)
        close(one[1:2], ref + blk.f64(bits(res)), abs_floor=2e-3)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)


@pytest.mark.parametrize("M,N,K", [(32, 4736, 520), (33, 4736, 520), (33, 4744, 520), (49, 4096, 4104), (64, 4736, 1032), (64, 128, 8), (48, 2048, 1000)])
def test_one_block_per_sm_from_33_rows(M, N, K):
    """Both sides of the line where few tiles (37 of 128 weight rows) take a whole SM's shared memory per block: against the oracle,
    rows around the output untouched."""
    x, w = rnd(M, K, seed=55), rnd(N, K, scale=K ** -0.5, seed=56)
    buf = torch.full((M + 2, N), 7.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear(x, w, buf[1:M + 1])
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    close(buf[1:M + 1], blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None), abs_floor=2e-3)
    assert torch.all(buf[0] == 7.0) and torch.all(buf[M + 1] == 7.0)


def test_a_refused_launch_is_reported_once():
    """2^40 rows make a grid of no blocks (2^32 cut to 32 bits), which the runtime refuses: that call says so, the next one, which looks at the
    runtime's last error behind its own launch, does not."""
    x, out = rnd(8, 16, seed=91), torch.empty(8, 8, dtype=torch.bfloat16, device="cuda")
    st = B().lib().relaxkv_swiglu(x.data_ptr(), out.data_ptr(), 1 << 40, 8, torch.cuda.current_stream().cuda_stream)
    assert st == B().ERR_CUDA
    scores = torch.ones(1, 64, device="cuda")
    B().relaxkv_scale_scores(B().Shape(8, 2, 128, [64], [1]), 1, scores, 0.5)
    assert torch.all(scores == 0.5)


def test_linear_at_the_benchmark_shapes():
    """The projections at the sizes the repair loop runs them for the 32K Qwen3-14B-shaped stack: 18 000 active rows
    through a 5120 -> 5120 projection with residual (SM pairs) and the fused gate/up projection of 5120 -> 2 x 17408 on
    2 000 rows; 128 rows (the query's prefill) and one row (a decode token) through the same weights.  Sampled
    rows against the oracle, every element against torch's fp32 matmul of the same bf16 inputs."""
    rng = np.random.default_rng(2)
    w = rnd(5120, 5120, scale=5120 ** -0.5, seed=71)
    for M in (18000, 128, 1):
        x, r = rnd(M, 5120, seed=72), rnd(M, 5120, seed=73)
        y = torch.full((M, 5120), 7.0, dtype=torch.bfloat16, device="cuda")
        B().relaxkv_linear(x, w, y, residual=r)
        st, detail = B().relaxkv_read_device_status()
        assert st == 0, (st, detail)
        torch.testing.assert_close(y.float(), x.float() @ w.float().T + r.float(), rtol=2e-2, atol=3e-2)
        rows = np.unique(rng.integers(0, M, size=min(M, 24)))
        idx = torch.from_numpy(rows).cuda()
        ref = blk.linear(blk.f64(bits(x[idx])), blk.f64(bits(w)), blk.f64(bits(r[idx])))
        close(y[idx], ref, abs_floor=4e-3)
    wgu = rnd(2 * 17408, 5120, scale=5120 ** -0.5, seed=74)
    tiled = B().tile_gate_up(wgu)
    for M in (2000, 128, 1):
        x = rnd(M, 5120, seed=75)
        out = torch.full((M, 17408), 7.0, dtype=torch.bfloat16, device="cuda")
        B().relaxkv_linear_swiglu(x, tiled, out)
        st, detail = B().relaxkv_read_device_status()
        assert st == 0, (st, detail)
        rows = np.unique(rng.integers(0, M, size=min(M, 12)))
        idx = torch.from_numpy(rows).cuda()
        ref = blk.swiglu(blk.linear(blk.f64(bits(x[idx])), blk.f64(bits(wgu)), None))
        close(out[idx], ref, abs_floor=4e-3)
        gu = x.float() @ wgu.float().T
        torch.testing.assert_close(out.float(), torch.nn.functional.silu(gu[:, :17408]) * gu[:, 17408:], rtol=2e-2, atol=3e-2)


def test_rmsnorm_rope_swiglu():
    # a few rows: one block per row; 4096 rows and more: whole rows through shared memory by bulk copies, also in place
    for rows, C in ((77, 640), (2500, 640), (4097, 640), (4100, 5120), (4099, 8192)):
        x, w = rnd(rows, C, seed=4, scale=3.0), rnd(C, seed=5)
        y = torch.empty_like(x)
        B().relaxkv_rmsnorm(x, w, y, 1e-6)
        ref = blk.rmsnorm(blk.f64(bits(x)), blk.f64(bits(w)), 1e-6)
        close(y, ref, abs_floor=1e-3)
        B().relaxkv_rmsnorm(x, w, x, 1e-6)
        close(x, ref, abs_floor=1e-3)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    for C in (64, 128, 256):                                    # head vectors: one warp per row, also in place
        xs, ws = rnd(53 * 5, C, seed=8, scale=2.0), rnd(C, seed=9)
        ref = blk.rmsnorm(blk.f64(bits(xs)), blk.f64(bits(ws)), 1e-6)
        B().relaxkv_rmsnorm(xs, ws, xs, 1e-6)
        close(xs, ref, abs_floor=1e-3)
    for D in (64, 128):
        q = rnd(53, 5, D, seed=6)
        pos = torch.tensor(np.random.default_rng(0).integers(0, 66000, size=53).astype(np.int32)).cuda()
        ref = blk.rope(blk.f64(bits(q)), pos.cpu().numpy(), 1e6)
        B().relaxkv_rope(q, pos, 1e6)
        close(q, ref, abs_floor=2e-3)
    gu = rnd(41, 2 * 264, seed=7, scale=2.0)
    out = torch.empty(41, 264, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_swiglu(gu, out)
    close(out, blk.swiglu(blk.f64(bits(gu))), abs_floor=1e-3)


@pytest.mark.parametrize("C", [264, 2048, 8192, 8200, 12288])
def test_rmsnorm_forms_at_their_line(C):
    """One block per row with the row in registers (up to 296 rows, 8192 columns held) and without (297): against the oracle, the same
    bits for a row in both, in place too."""
    x, w = rnd(297, C, seed=14, scale=2.0), rnd(C, seed=15)
    ys = []
    for rows in (297, 296):
        y = torch.full((298, C), 7.0, dtype=torch.bfloat16, device="cuda")
        B().relaxkv_rmsnorm(x[:rows], w, y[:rows], 1e-6)
        assert torch.all(y[rows:] == 7.0)
        z = x[:rows].clone()
        B().relaxkv_rmsnorm(z, w, z, 1e-6)
        assert torch.equal(z, y[:rows])
        ys.append(y)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    assert torch.equal(ys[0][:296], ys[1][:296])
    close(ys[0][:297], blk.rmsnorm(blk.f64(bits(x)), blk.f64(bits(w)), 1e-6), abs_floor=1e-3)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("with_norm", [True, False])
@pytest.mark.parametrize("n,H,Hkv", [(37, 5, 2), (2100, 40, 8), (2050, 18, 3), (4100, 40, 8), (4097, 18, 3)],
                         ids=["few_rows", "2100_rows_48_heads", "2050_rows_21_heads", "4100_rows_48_heads", "4097_rows_21_heads"])
def test_qk_norm_rope_in_one_launch(D, with_norm, n, H, Hkv):
    """Per-head RMSNorm (optional) + rotary embedding of q and k in one launch against the oracle's rmsnorm -> bf16
    storage -> rope per tensor, and against the library's own separate calls (equal up to the last bf16 bit of the
    normalised values); neighbouring rows untouched.  A few rows: four heads per block; 2048 rows and more: a block
    walks all heads of its row, four per warp in flight (48 heads: three batches for every warp; 21: a ragged one);
    4096 rows and more: one row per warp through shared memory by bulk copies, one head per half-warp (21 heads: the
    last pair is half empty)."""
    theta, eps = 1e6, 1e-6
    qb, kb = rnd(n + 2, H, D, seed=31, scale=2.0), rnd(n + 2, Hkv, D, seed=32, scale=2.0)
    q0, k0 = qb.clone(), kb.clone()
    wq, wk = (rnd(D, seed=33), rnd(D, seed=34)) if with_norm else (None, None)
    pos = torch.tensor(np.random.default_rng(1).integers(0, 70000, size=n).astype(np.int32)).cuda()
    q, k = qb[1:n + 1], kb[1:n + 1]
    B().relaxkv_qk_norm_rope(q, k, pos, theta, wq, wk, eps)
    for got, x0, w, heads in ((q, q0[1:n + 1], wq, H), (k, k0[1:n + 1], wk, Hkv)):
        x = blk.f64(bits(x0))
        if with_norm:
            x = bf16_round(blk.rmsnorm(x.reshape(n * heads, D), blk.f64(bits(w)), eps)).reshape(n, heads, D)
        ref = blk.rope(x, pos.cpu().numpy(), theta)
        # with the norm, the values are rounded to bf16 between the two steps on both sides; where fp32 and fp64 land on
        # different sides of a rounding tie, an input of the rotation moves by one bf16 ulp (2^-8 relative, of the
        # larger of the pair), which the small outputs inherit: the floor scales with the largest magnitude
        close(got, ref, abs_floor=max(4e-3, 2.0 ** -7 * float(np.abs(ref).max())) if with_norm else 2e-3)
        two = x0.clone()
        if with_norm:
            B().relaxkv_rmsnorm(two.view(-1, D), w, two.view(-1, D), eps)
        B().relaxkv_rope(two, pos, theta)
        assert float((two.float() - got.float()).abs().max()) <= 2.0 ** -6 * float(two.float().abs().max())
    assert torch.equal(qb[0], q0[0]) and torch.equal(qb[n + 1], q0[n + 1]) and torch.equal(kb[0], k0[0]) and torch.equal(kb[n + 1], k0[n + 1])


@pytest.mark.parametrize("ctx,chunk,C", [((640, 900), 128, 72), ((7000, 9500), 512, 1024)], ids=["few_rows", "many_rows"])
def test_target_positions_and_row_carry(ctx, chunk, C):
    """Positions of the targets and the carry of the rows that stay active, bit for bit; with some thousand rows the
    carry moves whole rows through shared memory by bulk copies."""
    from tests.harness import Case
    w = inputs.scaled_down(inputs.qwen14b_32k("calibrated"), ctx, (9, 17), n_layers=3, chunk=chunk)
    case = Case(w)
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    n_u, n_r = s.counts()
    if ctx[0] > 4096:
        assert sum(n_r[1]) >= 4096                      # the bulk form is the one under test
    for l in range(w.n_layers):
        total = sum(n_r[l])
        pos = torch.full((total,), -1, dtype=torch.int32, device="cuda")
        B().relaxkv_target_positions(s.shape, s.u_pos, s.u_cu, s.r_rank, s.r_cu_layer(l), n_r[l], pos)
        ref = np.concatenate([case.sets[b].positions(l) for b in range(w.n_req)])
        np.testing.assert_array_equal(pos.cpu().numpy(), ref)
        if l + 1 < w.n_layers:
            h = rnd(total, C, seed=10 + l)
            nxt = sum(n_r[l + 1])
            out = torch.zeros(nxt, C, dtype=torch.bfloat16, device="cuda")
            B().relaxkv_carry_rows(s.shape, h, out, s.r_rank, s.r_cu_layer(l), s.r_cu_layer(l + 1), n_r[l + 1])
            off = 0
            refs = []
            for b in range(w.n_req):
                hb = blk.f64(bits(h[off:off + n_r[l][b]]))
                refs.append(blk.compact_rows(hb, case.sets[b].ranks(l), case.sets[b].ranks(l + 1)))
                off += n_r[l][b]
            np.testing.assert_array_equal(out.float().cpu().numpy().astype(np.float64), np.concatenate(refs))
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)


def bf16_round(x: np.ndarray) -> np.ndarray:
    """Round float64 values to bf16 (nearest even) and return them as float64 - the storage precision of
    every tensor that travels between two kernels."""
    t = torch.from_numpy(np.ascontiguousarray(x)).to(torch.float32).to(torch.bfloat16)
    return t.to(torch.float64).numpy()


def to_bits(x: np.ndarray) -> np.ndarray:
    return inputs.bf16_bits(torch.from_numpy(np.ascontiguousarray(x)).to(torch.float32).to(torch.bfloat16))


def test_whole_repair_loop_with_block_work():
    """Algorithm 1, steps 13-22, three layers: the CUDA layer loop against the oracle chain.  The reference
    rounds every tensor that the GPU stores in bf16 to bf16 at the same points (storage precision is part of
    the data path); inside an operation it stays fp64."""
    from paper_2609_33503_b200.layer_loop import LayerLoop
    from tests.harness import Case
    w = inputs.Workload("block", 3, 4, 2, 64, 64, (600, 380), (8, 5), 0.15, base_seed=3,
                        planted_chunks=((2, 7), (1,)), variant="calibrated")
    blkshape = inputs.BlockShape(hidden=256, inter=512, rope_theta=1.0e4, eps=1.0e-5, qk_norm=True)
    case = Case(w)
    s = case.make_session()
    s.build_active_sets(case.anchors_tensor())
    n_u, n_r = s.counts()
    weights = [inputs.block_weights(w, blkshape, l, "cuda") for l in range(w.n_layers)]
    h0 = torch.cat([inputs.input_representations(w, blkshape, b, torch.from_numpy(case.sets[b].u_pos.astype(np.int64)), "cuda")
                    for b in range(w.n_req)]).contiguous()
    k_gpu = [k.clone() for k in case.k_cache]
    v_gpu = [v.clone() for v in case.v_cache]
    views = [B().CacheView(k, v, [int(x) for x in case.ctx_cu[:-1]]) for k, v in zip(k_gpu, v_gpu)]
    loop = LayerLoop(s, blkshape, sum(n_u))
    taps = []
    h_gpu = loop.run(h0, weights, views, taps=taps)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)

    # ---- one layer at a time: the oracle's block on the very rows the GPU layer received, so nothing compounds; a
    # wrong residual, a swapped norm gain or a missed projection cannot hide inside an end-to-end bound ----
    H, Hkv, D = w.n_q_heads, w.n_kv_heads, w.head_dim
    for l in range(w.n_layers):
        W = {k_: blk.f64(bits(v_)) for k_, v_ in weights[l].items()}
        h_in_all, h_out_all = taps[l]
        off = 0
        for b in range(w.n_req):
            sets = case.sets[b]
            pos = sets.positions(l)
            n = len(pos)
            h = blk.f64(bits(h_in_all[off:off + n]))
            x = bf16_round(blk.rmsnorm(h, W["w_in_norm"], blkshape.eps))
            q = bf16_round(blk.linear(x, W["wq"])).reshape(n, H, D)
            k = bf16_round(blk.linear(x, W["wk"])).reshape(n, Hkv, D)
            v = bf16_round(blk.linear(x, W["wv"])).reshape(n, Hkv, D)
            q = bf16_round(blk.rmsnorm(q.reshape(n * H, D), W["w_q_norm"], blkshape.eps)).reshape(n, H, D)
            k = bf16_round(blk.rmsnorm(k.reshape(n * Hkv, D), W["w_k_norm"], blkshape.eps)).reshape(n, Hkv, D)
            q, k = bf16_round(blk.rope(q, pos, blkshape.rope_theta)), bf16_round(blk.rope(k, pos, blkshape.rope_theta))
            o, _ = orc.repair_attention(case.req_k(l, b), case.req_v(l, b), to_bits(q), to_bits(k), to_bits(v), sets.u_pos,
                                        sets.ranks(l), case.scale)
            a = bf16_round(blk.linear(bf16_round(o).reshape(n, H * D), W["wo"], h))
            x2 = bf16_round(blk.rmsnorm(a, W["w_post_norm"], blkshape.eps))
            m = bf16_round(blk.swiglu(blk.linear(x2, W["w_gate_up"])))
            ref_l = bf16_round(blk.linear(m, W["w_down"], a))
            got_l = h_out_all[off:off + n].float().cpu().numpy().astype(np.float64)
            e = np.abs(got_l - ref_l)
            assert e.mean() <= 5e-3 * np.abs(ref_l).mean() and e.max() <= 0.06 * max(1.0, np.abs(ref_l).max()), \
                (l, b, e.mean() / np.abs(ref_l).mean(), e.max())
            off += n

    # ---- oracle chain, request by request ----
    off_u, final_refs = 0, []
    for b in range(w.n_req):
        sets = case.sets[b]
        h = blk.f64(bits(h0[off_u:off_u + len(sets.u_pos)]))
        off_u += len(sets.u_pos)
        for l in range(w.n_layers):
            W = {k_: blk.f64(bits(v_)) for k_, v_ in weights[l].items()}
            pos = sets.positions(l)
            n = len(pos)
            x = bf16_round(blk.rmsnorm(h, W["w_in_norm"], blkshape.eps))
            q = bf16_round(blk.linear(x, W["wq"])).reshape(n, H, D)
            k = bf16_round(blk.linear(x, W["wk"])).reshape(n, Hkv, D)
            v = bf16_round(blk.linear(x, W["wv"])).reshape(n, Hkv, D)
            q = bf16_round(blk.rmsnorm(q.reshape(n * H, D), W["w_q_norm"], blkshape.eps)).reshape(n, H, D)
            k = bf16_round(blk.rmsnorm(k.reshape(n * Hkv, D), W["w_k_norm"], blkshape.eps)).reshape(n, Hkv, D)
            q, k = bf16_round(blk.rope(q, pos, blkshape.rope_theta)), bf16_round(blk.rope(k, pos, blkshape.rope_theta))
            o, _ = orc.repair_attention(case.req_k(l, b), case.req_v(l, b), to_bits(q), to_bits(k), to_bits(v), sets.u_pos,
                                        sets.ranks(l), case.scale)
            o = bf16_round(o).reshape(n, H * D)
            # cache update: the GPU's repaired cache rows hold (its own) k, v of this layer
            lo = int(case.ctx_cu[b])
            gk = k_gpu[l][lo + torch.from_numpy(pos.astype(np.int64)).cuda()].float().cpu().numpy()
            dk = np.abs(gk - k)          # single-ulp differences of earlier tensors propagate: ~1 % of |k| on average
            assert dk.max() <= 0.1 * max(1.0, np.abs(k).max()) and dk.mean() <= 1e-2 * np.abs(k).mean(), (l, dk.max(), dk.mean())
            a = bf16_round(blk.linear(o, W["wo"], h))
            x2 = bf16_round(blk.rmsnorm(a, W["w_post_norm"], blkshape.eps))
            m = bf16_round(blk.swiglu(bf16_round(blk.linear(x2, W["w_gate_up"]))))
            h_out = bf16_round(blk.linear(m, W["w_down"], a))
            h = blk.compact_rows(h_out, sets.ranks(l), sets.ranks(l + 1)) if l + 1 < w.n_layers else h_out
        final_refs.append(h)
    ref = np.concatenate(final_refs)
    got = h_gpu.float().cpu().numpy().astype(np.float64)
    assert got.shape == ref.shape
    err = np.abs(got - ref)
    scale_ = np.abs(ref).mean()
    # three layers of bf16 tensors: single-ulp differences (fp32 vs fp64 accumulation) propagate, nothing more
    assert err.mean() <= 1e-2 * scale_ and err.max() <= 0.15 * max(1.0, np.abs(ref).max()), (err.mean(), err.max(), scale_)


@pytest.mark.parametrize("M,I,K", [(300, 256, 320), (129, 128, 72), (1000, 1024, 512), (1, 128, 8)])
def test_linear_swiglu_fused(M, I, K):
    """Gate and up projections + SwiGLU in one kernel (weights re-ordered per 128-feature block) against the
    oracle's linear followed by swiglu on the original [gate; up] weights."""
    x, w = rnd(M, K, seed=4), rnd(2 * I, K, scale=K ** -0.5, seed=5)
    out = torch.full((M, I), 7.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear_swiglu(x, B().tile_gate_up(w), out)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    ref = blk.swiglu(blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None))
    close(out, ref, abs_floor=2e-3)
    # the two-kernel route (projection rounded to bf16, then the activation) agrees to a rounding
    gu = torch.empty(M, 2 * I, dtype=torch.bfloat16, device="cuda")
    two = torch.empty_like(out)
    B().relaxkv_linear(x, w, gu)
    B().relaxkv_swiglu(gu, two)
    assert float((out.float() - two.float()).abs().max()) <= 2.0 ** -6 * float(two.float().abs().max()) + 1e-2


@pytest.mark.parametrize("M,I,K", [(96, 19072, 136), (97, 19072, 136), (128, 19072, 136), (128, 18944, 136), (2, 1024, 4096), (2, 3584, 4096), (2, 3712, 4096), (3, 1024, 4096), (4, 1024, 4104), (4, 1152, 4096), (3, 1024, 2048), (4, 2560, 5120)])
def test_gate_up_routes(M, I, K):
    """Both sides of the lines between the streaming kernel, the few-row tiles and the large kernel for gate/up matrices: against the oracle."""
    x, w = rnd(M, K, seed=57), rnd(2 * I, K, scale=K ** -0.5, seed=58)
    buf = torch.full((M + 2, I), 7.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear_swiglu(x, B().tile_gate_up(w), buf[1:M + 1])
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)
    close(buf[1:M + 1], blk.swiglu(blk.linear(blk.f64(bits(x)), blk.f64(bits(w)), None)), abs_floor=2e-3)
    assert torch.all(buf[0] == 7.0) and torch.all(buf[M + 1] == 7.0)


def test_rope_realigns_keys_of_a_moved_chunk():
    """Positional consistency (Section 2): a chunk cached at one offset and placed at another is re-aligned by
    rotating its cached keys by the offset difference.  The keys of a 512-token chunk are rotated at offset
    4096, then shifted by +8192 and by -3072 with the same kernel (positions = the delta for every token);
    the result must equal the oracle's rotation at the final positions."""
    T, Hkv, D, theta = 512, 8, 128, 1.0e6
    k_raw = rnd(T, Hkv, D, seed=21)
    old = torch.arange(4096, 4096 + T, dtype=torch.int32, device="cuda")
    for delta in (8192, -3072):
        k = k_raw.clone()
        B().relaxkv_rope(k, old, theta)                                               # the cached, chunk-time rotation
        B().relaxkv_rope(k, torch.full((T,), delta, dtype=torch.int32, device="cuda"), theta)   # re-alignment
        ref = blk.rope(blk.f64(bits(k_raw)), (old.cpu().numpy().astype(np.int64) + delta), theta)
        # two bf16 roundings instead of one
        g = k.float().cpu().numpy().astype(np.float64)
        assert np.all(np.abs(g - ref) <= 2.0 ** -7 * np.abs(ref) + 2e-2), float(np.abs(g - ref).max())
        # and attention logits against a query at a fixed position keep their relative-offset meaning
        q = rnd(1, Hkv, D, seed=22)
        qpos = torch.tensor([4096 + delta + T], dtype=torch.int32, device="cuda")
        B().relaxkv_rope(q, qpos, theta)
        logits = (q.float()[0][None] * k.float()).sum(-1).cpu().numpy()               # [T, Hkv]
        q_ref = blk.rope(blk.f64(bits(rnd(1, Hkv, D, seed=22))), qpos.cpu().numpy(), theta)
        ref_logits = (q_ref[0][None] * ref).sum(-1)
        assert np.abs(logits - ref_logits).max() <= 0.02 * np.sqrt(D) + 0.05 * np.abs(ref_logits).max()
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)


def test_query_pass_prefill_scores_and_first_decode_step():
    """The query's forward pass over [context cache, its own tokens] and one decode step (query_pass.QueryPass), two
    requests, two layers, synthetic weights, against the oracle one layer at a time on the rows the GPU layer received:
    the block chain of `relaxkv_block_oracle.decoder_block` with bf16 storage, causal attention by the oracle over the
    context rows plus the appended query K/V, the context scores of that very pass (supplied-normaliser scores), the
    K/V rows the pass appended to the cache, and the logits of the output head."""
    from paper_2609_33503_b200.query_pass import QueryPass
    H, Hkv, D = 4, 2, 64
    ctx, qn = (300, 170), (9, 5)
    blkshape = inputs.BlockShape(hidden=256, inter=512, rope_theta=1.0e4, eps=1.0e-5, qk_norm=True)
    w = inputs.Workload("qpass", 2, H, Hkv, D, 64, ctx, qn, 0.15, base_seed=11, planted_chunks=((1,), (0,)))
    L, nb, scale, vocab = 2, 2, D ** -0.5, 1000
    room = [c + q + 1 for c, q in zip(ctx, qn)]
    offs = [0, room[0] + 7]
    rows = offs[1] + room[1]
    weights = [inputs.block_weights(w, blkshape, l, "cuda") for l in range(L)]
    k_gpu, v_gpu, views = [], [], []
    for l in range(L):
        k_all = torch.zeros(rows, Hkv, D, dtype=torch.bfloat16, device="cuda")
        v_all = torch.zeros_like(k_all)
        for b in range(nb):
            _, k, v = inputs.layer_qkv(w, l, b, "cuda")
            k_all[offs[b]:offs[b] + ctx[b]], v_all[offs[b]:offs[b] + ctx[b]] = k, v
        k_gpu.append(k_all); v_gpu.append(v_all)
        views.append(B().CacheView(k_all, v_all, offs))
    k_ctx = [inputs.bf16_bits(k) for k in k_gpu]            # host copies of the context rows, before the pass appends to them
    v_ctx = [inputs.bf16_bits(v) for v in v_gpu]
    h0 = rnd(sum(qn), blkshape.hidden, seed=31)
    qp = QueryPass(H, Hkv, D, ctx, qn, blkshape, softmax_scale=scale)
    scores = torch.zeros(L, sum(ctx), dtype=torch.float32, device="cuda")
    taps = []
    h_last = qp.prefill(h0, weights, views, scores_out=scores, taps=taps)
    st, detail = B().relaxkv_read_device_status()
    assert st == 0, (st, detail)

    def check_layer(l, h_in_all, h_out_all, lens, pos0, k_rows, v_rows, want_scores):
        W = {k_: blk.f64(bits(v_)) for k_, v_ in weights[l].items() if k_ != "w_gate_up_tiled"}
        off = off_t = 0
        for b in range(nb):
            n = lens[b]
            pos = np.arange(pos0[b], pos0[b] + n)
            seen = {}

            def attend(q, k, v):
                kb = np.concatenate([k_rows[b], to_bits(k)])
                vb = np.concatenate([v_rows[b], to_bits(v)])
                seen.update(k=k, v=v, kb=kb, q=to_bits(q))
                o, lse = orc.list_attention(kb, vb, to_bits(q), None, None, np.arange(pos0[b] + n), pos, scale)
                seen["lse"] = lse
                return o

            ref = blk.decoder_block(blk.f64(bits(h_in_all[off:off + n])), W, H, Hkv, D, pos, blkshape.eps, blkshape.rope_theta,
                                    attend, store=bf16_round)
            got = h_out_all[off:off + n].float().cpu().numpy().astype(np.float64)
            e = np.abs(got - ref)
            assert e.mean() <= 5e-3 * np.abs(ref).mean() and e.max() <= 0.06 * max(1.0, np.abs(ref).max()), (l, b, e.mean(), e.max())
            # the K/V rows the pass appended to the cache (single-ulp differences of x propagate)
            gk = k_gpu[l][offs[b] + pos0[b]:offs[b] + pos0[b] + n].float().cpu().numpy()
            dk = np.abs(gk - seen["k"])
            assert dk.max() <= 0.1 * max(1.0, np.abs(seen["k"]).max()) and dk.mean() <= 1e-2 * np.abs(seen["k"]).mean()
            if want_scores:
                T = ctx[b]
                ref_raw = orc.raw_scores(seen["q"], seen["kb"][:T], scale, lse=seen["lse"].T)
                got_raw = scores[l, off_t:off_t + T].cpu().numpy().astype(np.float64)
                # the GPU's q differs from the oracle's by single ulps, which moves every logit a little: 2 % here, the
                # 1e-3 bound of the score kernel itself is tested on identical inputs elsewhere
                assert np.all(np.abs(got_raw - ref_raw) <= 2e-2 * ref_raw + 1e-5 / T), np.abs(got_raw / ref_raw - 1).max()
                off_t += T
            off += n

    for l in range(L):
        check_layer(l, taps[l][0], taps[l][1], qn, ctx, [k_ctx[l][offs[b]:offs[b] + ctx[b]] for b in range(nb)],
                    [v_ctx[l][offs[b]:offs[b] + ctx[b]] for b in range(nb)], True)

    # output head on the last query row of each request
    w_final, w_head = rnd(blkshape.hidden, seed=41), rnd(vocab, blkshape.hidden, scale=blkshape.hidden ** -0.5, seed=42)
    logits = torch.zeros(nb, vocab, dtype=torch.bfloat16, device="cuda")
    qp.output_head(h_last, w_final, w_head, logits)
    last = h_last[torch.tensor([qn[0] - 1, qn[0] + qn[1] - 1], device="cuda")]
    ref_logits = blk.output_head(blk.f64(bits(last)), blk.f64(bits(w_final)), blk.f64(bits(w_head)), blkshape.eps, store=bf16_round)
    close(logits, ref_logits, abs_floor=3e-2)

    # one decode step: a new token per request at position T_c + Q_b, one layer at a time as above
    k_after = [inputs.bf16_bits(k) for k in k_gpu]
    v_after = [inputs.bf16_bits(v) for v in v_gpu]
    h_tok = rnd(nb, blkshape.hidden, seed=51)
    for l in range(L):
        # run the decode of layer l alone on a known input row so that each layer is checked by itself
        out = qp.decode(h_tok, weights[l:l + 1], views[l:l + 1])
        st, detail = B().relaxkv_read_device_status()
        assert st == 0, (st, detail)
        check_layer(l, h_tok, out, (1, 1), [c + q for c, q in zip(ctx, qn)],
                    [k_after[l][offs[b]:offs[b] + ctx[b] + qn[b]] for b in range(nb)],
                    [v_after[l][offs[b]:offs[b] + ctx[b] + qn[b]] for b in range(nb)], False)


@pytest.mark.parametrize("graph", [False, True], ids=["eager", "graph"])
def test_decode_step_with_chained_launches_equals_plain_launches(graph):
    """The few-row kernels of a decode step are launched with programmatic stream serialization (each kernel's blocks
    become resident while its predecessor finishes and wait inside the kernel for it).  Same bits as plain launches:
    logits of three decode steps in a row and the K/V rows they append, eagerly and replayed from a CUDA graph."""
    from paper_2609_33503_b200.query_pass import QueryPass
    H, Hkv, D = 8, 2, 128
    ctx, qn = (700, 1300, 90), (1, 1, 1)
    blkshape = inputs.BlockShape(hidden=2048, inter=4096, rope_theta=1.0e6, eps=1.0e-6, qk_norm=True)
    w = inputs.Workload("chained", 3, H, Hkv, D, 64, ctx, qn, 0.15, base_seed=23)
    L, nb, vocab, steps = 3, 3, 3000, 3
    room = [c + q + steps for c, q in zip(ctx, qn)]
    offs = [0, room[0], room[0] + room[1]]
    weights = [inputs.block_weights(w, blkshape, l, "cuda") for l in range(L)]
    w_final, w_head = rnd(blkshape.hidden, seed=41), rnd(vocab, blkshape.hidden, scale=blkshape.hidden ** -0.5, seed=42)
    h_tok = rnd(nb, blkshape.hidden, seed=51)

    def run(chained):
        prev = B().relaxkv_set_chained_launch(chained)
        try:
            views, ks = [], []
            for l in range(L):
                k_all = torch.zeros(sum(room), Hkv, D, dtype=torch.bfloat16, device="cuda")
                v_all = torch.zeros_like(k_all)
                for b in range(nb):
                    _, k, v = inputs.layer_qkv(w, l, b, "cuda")
                    k_all[offs[b]:offs[b] + ctx[b]], v_all[offs[b]:offs[b] + ctx[b]] = k, v
                ks.append((k_all, v_all))
                views.append(B().CacheView(k_all, v_all, offs))
            qp = QueryPass(H, Hkv, D, ctx, qn, blkshape, extra_tokens=steps)
            logits = [torch.zeros(nb, vocab, dtype=torch.bfloat16, device="cuda") for _ in range(steps)]
            for s in range(steps):
                qp.decode_positions(s)

            def all_steps():
                for s in range(steps):
                    qp.output_head(qp.decode(h_tok, weights, views, step=s), w_final, w_head, logits[s])
            if graph:
                side = torch.cuda.Stream()
                side.wait_stream(torch.cuda.current_stream())
                with torch.cuda.stream(side):
                    all_steps()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=side):
                        all_steps()
                torch.cuda.current_stream().wait_stream(side)
                for lg in logits:
                    lg.zero_()
                g.replay()
            else:
                all_steps()
            torch.cuda.synchronize()
            st, detail = B().relaxkv_read_device_status()
            assert st == 0, (st, detail)
            return [lg.clone() for lg in logits], [(k.clone(), v.clone()) for k, v in ks]
        finally:
            B().relaxkv_set_chained_launch(prev)

    plain, chained = run(False), run(True)
    for s in range(steps):
        assert torch.isfinite(plain[0][s].float()).all() and plain[0][s].float().abs().max() > 0
        assert torch.equal(plain[0][s], chained[0][s]), s
    for (k0, v0), (k1, v1) in zip(plain[1], chained[1]):
        assert torch.equal(k0, k1) and torch.equal(v0, v1)
    # the appended rows are where they belong: position T_c + Q_b + step of every request is no longer zero
    for b in range(nb):
        for s in range(steps):
            assert plain[1][0][0][offs[b] + ctx[b] + qn[b] + s].float().abs().max() > 0


@pytest.mark.parametrize("layers", [7, 8, 9])
def test_scores_of_several_layers_in_one_launch_equal_the_layers_own(layers):
    """A query pass scores groups of eight layers behind the last of each where the rows of scores_out are one matrix, and each layer in
    its own launch where they are not: the same hidden rows, and scores that differ by the order of their fp32 sums alone (a
    column sum adds H * Q_b = 112 positive terms in at most 2 H_kv runs: 112 * 2^-24 < 1e-5 relative)."""
    from paper_2609_33503_b200.query_pass import QueryPass
    H, Hkv, D = 8, 2, 64
    ctx, qn = (700, 129), (9, 5)
    blkshape = inputs.BlockShape(hidden=256, inter=512, rope_theta=1.0e4, eps=1.0e-5, qk_norm=True)
    w = inputs.Workload("grouped", layers, H, Hkv, D, 64, ctx, qn, 0.15, base_seed=13)
    room = [c + q for c, q in zip(ctx, qn)]
    weights = [inputs.block_weights(w, blkshape, l, "cuda") for l in range(layers)]
    h0 = rnd(sum(qn), blkshape.hidden, seed=3)
    qp = QueryPass(H, Hkv, D, ctx, qn, blkshape)
    assert qp.q_kept.shape[0] == 8
    got = []
    for width in (sum(ctx), sum(ctx) + 4):                  # one matrix; rows with a gap between them
        views = [B().CacheView(rnd(sum(room), Hkv, D, seed=100 + l), rnd(sum(room), Hkv, D, seed=200 + l), [0, room[0]]) for l in range(layers)]
        scores = torch.full((layers, width), -1.0, dtype=torch.float32, device="cuda")[:, :sum(ctx)]
        h = qp.prefill(h0, weights, views, scores_out=scores)
        st, detail = B().relaxkv_read_device_status()
        assert st == 0, (st, detail)
        got.append((h.clone(), scores.contiguous()))
    assert torch.equal(got[0][0], got[1][0])
    assert (got[1][1] > 0).all()
    assert ((got[0][1] - got[1][1]).abs() <= 1e-5 * got[1][1]).all()


@pytest.mark.parametrize("head_major", [False, True], ids=["token_major", "head_major"])
@pytest.mark.parametrize("H,Hkv,D,with_norm,counts", [(4, 1, 64, False, (1,)), (6, 2, 128, True, (1, 0, 7)), (40, 8, 128, True, (130,)), (8, 8, 64, True, (256, 257))],
                         ids=["one_row", "ragged", "query", "two_launches"])
def test_rotating_and_appending_in_one_launch(H, Hkv, D, with_norm, counts, head_major):
    """relaxkv_qk_norm_rope_append: the bits of relaxkv_qk_norm_rope followed by relaxkv_scatter_kv_lists, in q, k and the cache (513 rows:
    more than one launch takes); rows past a request's host bound or at a position outside it are reported and appended nowhere."""
    n, nb = sum(counts), len(counts)
    ctx = [300 + 11 * b for b in range(nb)]
    offs = [sum(ctx[:b]) + 5 * b for b in range(nb)]
    rows = offs[-1] + ctx[-1]
    rng = np.random.default_rng(n)
    pos = torch.from_numpy(np.concatenate([np.sort(rng.choice(c, m, replace=False)) for c, m in zip(ctx, counts)]).astype(np.int32)).cuda()
    cu = torch.tensor([sum(counts[:b]) for b in range(nb + 1)], dtype=torch.int32, device="cuda")
    wq, wk = (rnd(D, seed=3), rnd(D, seed=4)) if with_norm else (None, None)
    shape = B().Shape(H, Hkv, D, ctx)

    def run(fn, pos, bounds):
        q, k, v = rnd(n, H, D, seed=5), rnd(n, Hkv, D, seed=6), rnd(n, Hkv, D, seed=7)
        kv = [rnd(Hkv, rows, D, seed=8 + i).transpose(0, 1) if head_major else rnd(rows, Hkv, D, seed=8 + i) for i in range(2)]
        fn(B().CacheView(kv[0], kv[1], offs), q, k, v, pos, bounds)
        return [t.clone() for t in (q, k, *kv)], B().relaxkv_read_device_status()[0]

    def two(cache, q, k, v, pos, bounds):
        B().relaxkv_qk_norm_rope(q, k, pos, 1e6, wq, wk, 1e-6)
        B().relaxkv_scatter_kv_lists(shape, cache, k, v, pos, cu, bounds)

    def one(cache, q, k, v, pos, bounds):
        B().relaxkv_qk_norm_rope_append(shape, cache, q, k, v, pos, cu, bounds, 1e6, wq, wk, 1e-6)

    outside = pos.clone()
    outside[-1] = ctx[-1]
    for p, bounds in ((pos, counts), (outside, counts), (pos, [max(0, c - 1) for c in counts])):
        (want, st2), (got, st1) = run(two, p, bounds), run(one, p, bounds)
        assert all(torch.equal(a, b) for a, b in zip(want, got))
        assert st1 == st2 and (st1 != 0) == (p is outside or (bounds is not counts and any(bounds)))


@pytest.mark.parametrize("M", [129, 300, 1000])
@pytest.mark.parametrize("N,off_y,off_r", [(512, 0, 0), (512, 8, 0), (512, 0, 8), (264, 0, 0), (272, 8, 8), (8, 0, 0)])
def test_rows_of_any_alignment_leave_a_gemm_alike(M, N, off_y, off_r):
    """Both GEMM kernels store (and add) whole 32-byte sectors where every row is 32-byte aligned and 16-byte pieces elsewhere: the same bits
    as an aligned output of a width of 512, neighbours untouched."""
    K = 192
    x, w, r = rnd(M, K, seed=1), rnd(512, K, scale=K ** -0.5, seed=2), rnd(M, 512, seed=3)
    ref = torch.empty(M, 512, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear(x, w, ref, residual=r)
    res = torch.zeros(M * N + 16, dtype=torch.bfloat16, device="cuda")
    res[off_r:off_r + M * N] = r[:, :N].reshape(-1)
    out = torch.full((M * N + 16,), 3.0, dtype=torch.bfloat16, device="cuda")
    B().relaxkv_linear(x, w[:N].contiguous(), out[off_y:off_y + M * N].view(M, N), residual=res[off_r:off_r + M * N].view(M, N))
    assert torch.equal(out[off_y:off_y + M * N].view(M, N), ref[:, :N])
    assert torch.all(out[:off_y] == 3.0) and torch.all(out[off_y + M * N:] == 3.0)


def _grouped_pass(layers=3):
    """A small query pass with scores: the pass, weights, query rows, per-layer K/V, a view of a layer's tensors, its scores by single layers."""
    from paper_2609_33503_b200.query_pass import QueryPass
    H, Hkv, D, ctx, qn = 8, 2, 64, (700,), (9,)
    blkshape = inputs.BlockShape(hidden=256, inter=512, rope_theta=1.0e4, eps=1.0e-5, qk_norm=True)
    w = inputs.Workload("staged", layers, H, Hkv, D, 64, ctx, qn, 0.15, base_seed=13)
    rows = ctx[0] + qn[0]
    weights = [inputs.block_weights(w, blkshape, l, "cuda") for l in range(layers)]
    kv = [(rnd(rows, Hkv, D, seed=100 + l), rnd(rows, Hkv, D, seed=200 + l)) for l in range(layers)]
    view = lambda k, v: B().CacheView(k, v, [0])
    qp, h0 = QueryPass(H, Hkv, D, ctx, qn, blkshape), rnd(qn[0], blkshape.hidden, seed=3)
    apart = torch.full((layers, ctx[0] + 4), -1.0, device="cuda")[:, :ctx[0]]            # rows with a gap: a launch per layer
    h = qp.prefill(h0, weights, [view(k.clone(), v.clone()) for k, v in kv], scores_out=apart).clone()
    return qp, weights, h0, kv, view, h, apart


class _Staged:
    """Caches that a program streams: asked for a layer, it copies that layer into the one staging buffer there is, and hands it out once."""

    def __init__(self, kv, view, n_buffers):
        self.kv, self.next = kv, 0
        self.views = [view(torch.empty_like(kv[0][0]), torch.empty_like(kv[0][1])) for _ in range(n_buffers)]

    def __len__(self):
        return len(self.kv)

    def __getitem__(self, l):
        assert l == self.next, "a layer that was handed out, or is not due yet"
        self.next += 1
        c = self.views[l % len(self.views)]
        c.k.copy_(self.kv[l][0])
        c.v.copy_(self.kv[l][1])
        return c


@pytest.mark.parametrize("n_buffers", [1, 2])
@pytest.mark.parametrize("by", ["sequence", "weights"])
def test_scores_of_a_pass_whose_caches_are_staged(by, n_buffers):
    """One or two staging buffers for the caches of all layers, filled when a layer is asked for, or by the generator of the layers' weights
    (which has no length): every layer's scores are its own, to the order of fp32 sums (112 positive terms at most: 1e-5)."""
    qp, weights, h0, kv, view, h_ref, ref = _grouped_pass()
    staged, scores = _Staged(kv, view, n_buffers), torch.full(ref.shape, -1.0, device="cuda")
    if by == "sequence":
        h = qp.prefill(h0, weights, staged, scores_out=scores)
    else:
        def stream():
            for l, w in enumerate(weights):
                staged[l]
                yield w
        h = qp.prefill(h0, stream(), [staged.views[l % n_buffers] for l in range(len(weights))], scores_out=scores)
    assert B().relaxkv_read_device_status()[0] == 0
    assert torch.equal(h, h_ref)
    assert ((scores - ref).abs() <= 1e-5 * ref).all()


@pytest.mark.parametrize("layout", ["one_tensor", "interleaved", "same"])
def test_scores_of_a_pass_by_the_memory_of_its_layers(layout):
    """Layers whose caches are slices of one tensor, lie between one another's rows, or are one cache (each layer then sees the query rows
    of the layers before in the rows behind the context, which no score reads)."""
    qp, weights, h0, kv, view, h_ref, ref = _grouped_pass()
    L = len(kv)
    if layout == "same":
        kv = [kv[0]] * L
        views = [view(*kv[0])] * L
        ref = torch.cat([ref[:1]] * L)                   # (of layer 0 alone: the others' queries differ from the reference pass)
    else:
        stacked = [torch.stack([x[i] for x in kv], dim=0 if layout == "one_tensor" else 1) for i in range(2)]
        views = [view(*(t[l] if layout == "one_tensor" else t[:, l] for t in stacked)) for l in range(L)]
    scores = torch.full(ref.shape, -1.0, device="cuda")
    h = qp.prefill(h0, weights, views, scores_out=scores)
    assert B().relaxkv_read_device_status()[0] == 0
    n = 1 if layout == "same" else L
    assert ((scores[:n] - ref[:n]).abs() <= 1e-5 * ref[:n]).all() and (scores > 0).all()
    if layout != "same":
        assert torch.equal(h, h_ref)
