"""The graph build's sorts and pair index at the edges of their tiles: one exact count per view
order and the static edge count, against numpy, at sizes around a tile (4,096 edges), with one to
four digits of node ids, skewed and loop-ridden, for both time widths."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _count_two(src, dst, t, delta, kind):
    """Two-edge motifs by one pass over each node's (or pair's) time-sorted list."""
    by = {}
    n = 0
    for s, d, x in zip(src.tolist(), dst.tolist(), t.tolist()):
        if s == d:
            continue
        key = s if kind == "out" else d if kind == "in" else (s, d)
        other = d if kind == "out" else s
        for o, y in reversed(by.get(key, ())):
            if x - y > delta:
                break
            n += y < x and (kind == "pair" or o != other)
        by.setdefault(key, []).append((other, x))
    return n


@pytest.mark.parametrize("n_nodes", [1, 2, 33, 1_000, 1_030, 40_000, 1_100_000, 1_500_000_000])
@pytest.mark.parametrize("m", [1, 31, 4_095, 4_096, 4_097, 12_289])
def test_views_and_pairs_at_tile_edges(n_nodes, m):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    if n_nodes > 10**9 and m != 4_097:
        pytest.skip("offsets of 1.5e9 nodes: one size is enough")
    rng = np.random.default_rng(n_nodes % 1000 + m)
    # half the endpoints among a few hubs, the rest over the whole id range
    def ends():
        x = rng.integers(0, n_nodes, m)
        hub = rng.random(m) < 0.5
        x[hub] = (rng.integers(0, min(n_nodes, 5), int(hub.sum())) * 7919) % n_nodes
        x[-1] = n_nodes - 1
        return x.astype(np.int32)
    src, dst = ends(), ends()
    for step in (1, 1 << 40):   # 32-bit and 64-bit times
        t = np.sort(rng.integers(0, max(m // 2, 1), m)).astype(np.int64) * step
        delta = 40 * step
        with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), n_nodes) as g:
            assert g.info().n_pairs == len(set(zip(src.tolist(), dst.tolist())))
            for kind, (ms, md) in {"out": ([0, 0], [1, 2]), "in": ([1, 2], [0, 0]), "pair": ([0, 0], [1, 1])}.items():
                assert tm.count_exact(g, tm.Motif(ms, md), delta) == _count_two(src, dst, t, delta, kind), kind


def test_wrong_inputs_keep_their_order_of_blame():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    m = 5_000
    base = np.arange(m, dtype=np.int64)
    ids = (np.arange(m) % 7).astype(np.int32)

    def status(src, dst, t, n):
        with pytest.raises(tm.TmError) as e:
            tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), n)
        return e.value.status

    bad_t = base.copy()
    bad_t[4_500] = 3
    bad_id = ids.copy()
    bad_id[4_999] = 7
    far = base.copy()
    far[-1] = 1 << 61
    neg = ids.copy()
    neg[0] = -2
    assert status(ids, ids, bad_t, 7) == tm.TM_EUNSORTED
    assert status(bad_id, ids, bad_t, 7) == tm.TM_EUNSORTED
    assert status(ids, bad_id, base, 7) == tm.TM_ERANGE
    assert status(neg, ids, base, -1) == tm.TM_ERANGE
    assert status(ids, ids, base, 0) == tm.TM_ERANGE
    assert status(ids, ids, far, 7) == tm.TM_EINVAL
    assert status(bad_id, ids, far, 7) == tm.TM_ERANGE
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (ids, ids, base)), -1) as g:
        assert g.info().n_nodes == 7


@pytest.mark.parametrize("crowded", [False, True])
def test_pair_table_filled_by_parts(crowded):
    """A graph large enough for the pair table to be filled part by part, and one whose pairs all
    hash into a single part (more than its list holds): every reply pair is found."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    rng = np.random.default_rng(8)
    n, m = 20_000, (3 << 20) + 1
    u, v = rng.integers(0, n, 6_000_000), rng.integers(0, n, 6_000_000)
    if crowded:
        x = (u.astype(np.uint64) << np.uint64(32)) | v.astype(np.uint64)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x ^= x >> np.uint64(31)
        keep = np.flatnonzero((x >> np.uint64(58)) == 5)
        assert len(keep) > 80_000
        u, v = u[keep], v[keep]
        pick = rng.integers(0, len(u), m)
        src, dst = u[pick].astype(np.int32), v[pick].astype(np.int32)
    else:
        half = m // 2   # replies are common
        src = np.concatenate([u[:half], v[:m - half]]).astype(np.int32)
        dst = np.concatenate([v[:half], u[:m - half]]).astype(np.int32)
        order = rng.permutation(m)
        src, dst = src[order], dst[order]
    t = np.sort(rng.integers(0, 50_000, m)).astype(np.int64)
    delta, span = 20_000, 100_000
    pair = src.astype(np.int64) * n + dst
    keys = np.sort(pair * span + t)
    rev = (dst.astype(np.int64) * n + src) * span + t
    ok = src != dst
    want = int((np.searchsorted(keys, rev + delta, "right") - np.searchsorted(keys, rev, "right"))[ok].sum())
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), n) as g:
        assert g.info().n_pairs == len(np.unique(pair))
        assert tm.count_exact(g, tm.Motif([0, 1], [1, 0]), delta) == want
