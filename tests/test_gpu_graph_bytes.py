"""tm_graph_info.device_bytes: what the graph's arrays, its pair filter and its pair table take,
whichever way the table was built."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _up(x):
    return (x + 255) & ~255


def _expected(m, n, table):
    """Arrays of a graph with 32-bit times, the filter, and a table of `table` bytes."""
    words = 1
    while words < (m + 7) // 8 and words < 1 << 23:
        words <<= 1
    i32, off = _up(4 * m), _up(8 * (n + 1))
    return 3 * i32 + 2 * (off + 3 * i32) + 4 * i32 + 4 * words + table


def _pow2(need):
    x = 2
    while 2 * x < 3 * need:
        x <<= 1
    return x


def _crowd(u, v):
    """The pairs that fall into one list of the table's first step (SplitMix64, upper six bits)."""
    x = (u.astype(np.uint64) << np.uint64(32)) | v.astype(np.uint64)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return np.flatnonzero(((x ^ (x >> np.uint64(31))) >> np.uint64(58)) == 5)


@pytest.mark.parametrize("kind", ["inserted", "parts", "crowded", "few", "few and small"])
def test_device_bytes_count_the_table_that_is_there(kind):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    rng = np.random.default_rng(8)
    n, m = 20_000, {"inserted": 100_003, "few": 1_500_001, "few and small": 50_001}.get(kind, (1 << 21) + 5)
    u, v = rng.integers(0, n, 6_000_000), rng.integers(0, n, 6_000_000)
    u[50:100], v[50:100] = v[:50].copy(), u[:50].copy()   # (a few pairs with replies)
    pool = _crowd(u, v) if kind == "crowded" else np.arange(100 if kind.startswith("few") else len(u))
    pick = pool[rng.integers(0, len(pool), m)]
    src, dst = u[pick].astype(np.int32), v[pick].astype(np.int32)
    t = np.sort(rng.integers(0, 50_000, m)).astype(np.int64)
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), n) as g:
        info = g.info()
        pairs = len(np.unique(src.astype(np.int64) * n + dst))
        assert info.n_pairs == pairs
        if kind in ("inserted", "few and small"):
            table = 16 * _pow2(m)
        elif kind in ("crowded", "few"):   # by the pairs
            table = 16 * _pow2(pairs)
        else:
            table = 64 * -(-pairs // (64 * 1900)) * 4096 * 16
        assert info.device_bytes == _expected(m, n, table), (kind, info.device_bytes)
        # the table answers: replies within 3 ticks
        key = np.sort((src.astype(np.int64) * n + dst) * 100_000 + t)
        rev = ((dst.astype(np.int64) * n + src) * 100_000 + t)[src != dst]
        want = int((np.searchsorted(key, rev + 3, "right") - np.searchsorted(key, rev, "right")).sum())
        assert tm.count_exact(g, tm.Motif([0, 1], [1, 0]), 3) == want
