"""Estimates that share one enumeration no query asked for: each equals itself run alone, bit for
bit, and the oracle, for three and four edges, few and many riders, and both time widths (the
wider with 64-bit window indices and weights without a table)."""
import pytest

from paper_1810_00980_gb300 import synth

pytestmark = pytest.mark.gpu

KEYS = ("status", "count", "estimate", "windows", "windows_kept", "var_hat", "shift_var", "p_used")
MOTIFS = {
    "cycle3": ([0, 1, 2], [1, 2, 0]),
    "outstar3": ([2, 2, 2], [0, 1, 0]),
    "pingpong": ([0, 1, 0], [1, 0, 1]),
    "cycle4": ([0, 1, 2, 3], [1, 2, 3, 0]),      # closed from either side
    "square4": ([0, 1, 2, 0], [1, 2, 0, 1]),     # last edge repeats the first pair
    "tail4": ([0, 0, 1, 3], [1, 2, 3, 0]),       # last edge closes the newest node
}


@pytest.mark.parametrize("ticks,many", [(1, False), (1, True), (6000, True)])
@pytest.mark.parametrize("name", list(MOTIFS))
def test_shared_estimates_equal_alone(name, ticks, many):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    import oracle
    from paper_1810_00980_gb300 import tm
    src, dst, t = synth.chung_lu_hawkes(200, 9_000, 2.1, seed=13, horizon=400_000)
    t = t * ticks
    ms, md = MOTIFS[name]
    mo, d = tm.Motif(ms, md), 600 * ticks
    specs = [(d, 10, 0.8, 1, 1, 0), (d // 6, 5, 0.9, 2, 2, 0), (d, 30, 1.0, 3, 1, 0), (d, 1, 0.5, 4, 1, 0),
             (d // 2, 7, 40.0, 5, 2, 1)]
    if many:
        specs += [(d, 10 + s % 3, 0.1, 100 + s, 1, 0) for s in range(40)]
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), 200) as g:
        qs = [tm.estimate_query(mo, dl, c, p, s, b=b, q_mode=qm) for dl, c, p, s, b, qm in specs]
        res = tm.run_batch(g, qs)
        assert sum(r["first_edges"] > 0 for r in res) == 1     # one enumeration for all of them
        for q, r, (dl, c, p, s, b, qm) in zip(qs, res, specs):
            # alone: by itself for p below 1, the whole-graph pass for p = 1
            one = tm.run_batch(g, [q])[0]
            assert {k: r[k] for k in KEYS} == {k: one[k] for k in KEYS}, (dl, c, p, s)
            if qm == 0 and s < 102:
                want = oracle.estimate(src, dst, t, ms, md, dl, c, p, s, b=b, threads=4)
                assert abs(r["estimate"] - want) <= 1e-12 * max(abs(want), 1e-300) or r["estimate"] == want == 0
        # beside an exact query of the motif the same estimates ride along with that one
        both = tm.run_batch(g, [tm.exact_query(mo, d)] + qs)
        assert both[0]["count"] == oracle.count_exact(src, dst, t, ms, md, d, threads=4)
        assert [{k: r[k] for k in KEYS} for r in both[1:]] == [{k: r[k] for k in KEYS} for r in res]


def test_few_windows_stay_alone():
    """Sparse estimates keep their own enumeration (its counters are theirs)."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    src, dst, t = synth.chung_lu_hawkes(700, 40_000, 2.1, seed=13, horizon=2_000_000)
    mo = tm.Motif(*MOTIFS["cycle3"])
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), 700) as g:
        res = tm.run_batch(g, [tm.estimate_query(mo, 3600, 10, 0.2, s) for s in range(4)])
        assert all(r["first_edges"] > 0 for r in res)


def test_no_room_for_the_records_runs_the_estimates_apart():
    """The shared enumeration needs a record buffer that the estimates alone do not: when it
    cannot be had, the batch still runs and equals itself."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    src, dst, t = synth.chung_lu_hawkes(700, 40_000, 2.1, seed=13, horizon=2_000_000)
    mo = tm.Motif(*MOTIFS["cycle3"])
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), 700) as g:
        qs = [tm.estimate_query(mo, 3600, 10, 0.8, s) for s in range(3)]
        ref = tm.run_batch(g, qs)
        assert sum(r["first_edges"] > 0 for r in ref) == 1
        try:
            tm.set_ride_capacity(1 << 36)   # 1.6 TB of records
            res = tm.run_batch(g, qs)
        finally:
            tm.set_ride_capacity(1 << 23)
        assert all(r["first_edges"] > 0 for r in res)
        assert [{k: r[k] for k in KEYS} for r in res] == [{k: r[k] for k in KEYS} for r in ref]
        assert tm.run_batch(g, qs)[0]["estimate"] == ref[0]["estimate"]
