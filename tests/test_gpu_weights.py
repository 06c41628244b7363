"""The Q64 weight of one instance, bit for bit: floor(c delta 2^64 / (c delta - Delta)) through
the weight table and through the per-instance division, on both sides of a 32-bit divisor."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [
    # (delta, c, duration)
    (1, 1, 0), (7, 2, 7), (3600, 10, 3599), (86400, 30, 1),
    (4095, 1048576, 4000),            # c delta just below 2^32
    (4097, 1048576, 4097),            # divisor on the other side of 2^32
    (1000, 5_000_000, 999),           # 64-bit divisor, table
    ((1 << 22) - 1, 1, (1 << 22) - 2),   # the longest table
    (1 << 22, 3, 1 << 22),            # first span without one
    (86_400_000, 30, 86_399_999),     # 64-bit divisor, no table
    (1 << 40, 1 << 19, (1 << 40) - 1),
]


@pytest.mark.parametrize("delta,c,dur", CASES)
def test_weight_of_one_instance_is_exact(delta, c, dur):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    dur = max(dur, 1) if delta > 1 else dur
    # an instance of two edges dur ticks apart (dur = 0: an instance of one edge)
    if dur:
        src, dst, t, mo = [0, 1], [1, 2], [0, dur], tm.Motif([0, 1], [1, 2])
    else:
        src, dst, t, mo = [0], [1], [0], tm.Motif([0], [1])
    g = tm.Graph(np.array(src, np.int32), np.array(dst, np.int32), np.array(t, np.int64), 3)
    want = (c * delta << 64) // (c * delta - dur)
    seen = 0
    for seed in range(40):
        _, wins = tm.estimate_windows(g, mo, delta, c, 1.0, seed)
        got = sum((w["w_int"] << 64) + w["w_frac"] for w in wins)
        assert got in (0, want), (seed, got, want)
        seen += got == want
        # in a batch that shares the table with a query of the same spans
        rs = tm.run_batch(g, [tm.estimate_query(mo, delta, c, 1.0, seed)] * 3)
        assert all(r["count"] == (got == want) for r in rs)
        if got:
            assert all(abs(r["estimate"] - want / 2**64) <= 1e-12 * want / 2**64 for r in rs)
    if c > 1 and dur < c * delta // 2:
        assert seen   # the instance fits a window for most shifts
