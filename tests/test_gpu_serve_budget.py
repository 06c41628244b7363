"""A server whose budget has no room for a record buffer runs the estimates of a batch apart; with room
they share an enumeration.  Results are the same."""
import pytest

from paper_1810_00980_gb300 import synth

pytestmark = pytest.mark.gpu

KEYS = ("status", "count", "estimate", "windows_kept", "var_hat")


@pytest.mark.parametrize("budget", [64 << 20, 1 << 30])
def test_sharing_stays_inside_the_budget(budget):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    src, dst, t = synth.chung_lu_hawkes(700, 40_000, 2.1, seed=13, horizon=2_000_000)
    mo, four = tm.Motif(*synth.MOTIFS["cycle3"]), tm.Motif(*synth.MOTIFS["cycle4"])
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), 700) as g:
        qs = [tm.estimate_query(mo, 3600, 10, 0.8, s) for s in range(12)]
        want = [tm.run_batch(g, [q])[0] for q in qs]
        shared = False
        for _ in range(20):
            with tm.Server(n_streams=1, max_batch=64, mem_budget_bytes=budget) as srv:
                gid = srv.attach(g)
                srv.submit(gid, tm.exact_query(four, 86400))     # (the others queue up behind it)
                tickets = [srv.submit(gid, q) for q in qs]
                res = [srv.wait(x, 60_000)[1] for x in tickets]
            assert [{k: r[k] for k in KEYS} for r in res] == [{k: r[k] for k in KEYS} for r in want]
            if budget < 192 << 20:
                assert all(r["first_edges"] > 0 for r in res)
            shared |= any(r["first_edges"] == 0 for r in res)
            if shared:
                break
        assert shared == (budget >= 192 << 20)
