"""The repair schedule of one request in one launch (little work) and in four: the edges of its lists, bad anchors, where the counts go.
Integer work: bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import relaxkv_oracle as orc

pytestmark = pytest.mark.gpu


def B():
    from paper_2609_33503_b200 import binding
    return binding


def _session(T, L, k):
    from paper_2609_33503_b200.pipeline import RepairSession
    s = RepairSession(8, 2, 128, [T], [1], L, [k])
    for t in (s.highest_layer, s.u_pos, s.u_cu, s.u_rank, s.r_rank, s.r_cu, s.counts_pinned):
        t.fill_(-7)
    return s


def _anchors(rng, T, L, k):
    return np.stack([np.sort(rng.choice(T, size=k, replace=False)) for _ in range(L)]).astype(np.int32)


def _highest(anchors, T):
    h = np.full(T, -1, dtype=np.int32)
    for l, row in enumerate(anchors):
        h[row[(row >= 0) & (row < T)]] = l
    return h


def _check(s, h, counts):
    """Every output against the highest layers h, written out from their definition."""
    L = s.n_layers
    u = np.flatnonzero(h >= 0)
    np.testing.assert_array_equal(s.highest_layer.cpu().numpy(), h)
    np.testing.assert_array_equal(s.u_cu.cpu().numpy(), [0, len(u)])
    np.testing.assert_array_equal(s.u_pos[:len(u)].cpu().numpy(), u)
    rank = np.full(len(h), -1)
    rank[u] = np.arange(len(u))
    np.testing.assert_array_equal(s.u_rank.cpu().numpy(), rank)
    lists = [np.flatnonzero(h[u] >= l) for l in range(L)]
    np.testing.assert_array_equal(s.r_cu.cpu().numpy(), np.concatenate([[0], np.cumsum([len(r) for r in lists])]))
    np.testing.assert_array_equal(s.r_rank[:sum(map(len, lists))].cpu().numpy(), np.concatenate(lists))
    if counts is not None:
        assert counts.tolist() == [len(u)] + [len(r) for r in lists]


@pytest.mark.parametrize("T,L", [(1024, 15), (1024, 16), (1024, 31), (1024, 32), (1024, 33), (257, 100), (33, 254), (256, 255), (1, 40), (8192, 7), (8192, 8),
                                 (8193, 6), (65536, 1), (2048, 31), (2048, 32)])
def test_one_request(T, L):
    """16 lists and more are a warp's own, 33 and more give a warp several; 255 layers are the most of the one-launch form; slices x lists
    of 8192 are its last (8192 positions x 8 lists, 2048 x 32) and the next shape takes the four launches."""
    rng = np.random.default_rng(T + L)
    k = max(1, T // 7)
    a = _anchors(rng, T, L, k)
    s = _session(T, L, k)
    s.build_active_sets(torch.from_numpy(a).cuda())
    torch.cuda.synchronize()
    assert B().relaxkv_read_device_status()[0] == 0
    ref = orc.active_sets(a, T)
    h = _highest(a, T)
    np.testing.assert_array_equal(np.flatnonzero(h >= 0), ref.u_pos)
    _check(s, h, s.counts_pinned)


@pytest.mark.parametrize("T,L", [(1024, 3), (40000, 3)])
def test_anchor_out_of_range_is_reported_and_left_out(T, L):
    """-1 and T among the anchors: the status word says so, the schedule is the one of the other anchors, and what lies beside the outputs
    stays as it was."""
    rng = np.random.default_rng(5)
    k = T // 8
    a = _anchors(rng, T, L, k)
    a[0, 3], a[2, k - 1] = -1, T
    s = _session(T, L, k)
    guarded = {}
    for name in ("highest_layer", "u_rank"):
        buf = torch.full((T + 64,), -9, dtype=torch.int32, device="cuda")
        guarded[name] = buf
        setattr(s, name, buf[32:32 + T])
    s.build_active_sets(torch.from_numpy(a).cuda())
    torch.cuda.synchronize()
    st, _ = B().relaxkv_read_device_status()
    assert st == B().ERR_BAD_INDEX
    _check(s, _highest(a, T), s.counts_pinned)
    for buf in guarded.values():
        assert torch.all(buf[:32] == -9) and torch.all(buf[32 + T:] == -9)


@pytest.mark.parametrize("T", [1024, 40000])
@pytest.mark.parametrize("where", ["pageable", "absent", "pinned"])
def test_counts_go_where_the_caller_asks(T, where):
    rng = np.random.default_rng(6)
    L, k = 4, T // 9
    a = _anchors(rng, T, L, k)
    s = _session(T, L, k)
    counts = None if where == "absent" else torch.full((1 + L + 2,), -7, dtype=torch.int32, pin_memory=where == "pinned")
    d = torch.from_numpy(a).cuda()
    B().relaxkv_build_active_sets(s.shape, L, s.k, d, s.highest_layer, s.u_pos, s.u_cu, s.u_rank, s.r_rank, s.r_cu, s.workspace,
                                  counts_pinned=counts)
    torch.cuda.synchronize()
    assert B().relaxkv_read_device_status()[0] == 0
    _check(s, _highest(a, T), None if counts is None else counts[:1 + L])
    if counts is not None:
        assert counts[1 + L:].tolist() == [-7, -7]
