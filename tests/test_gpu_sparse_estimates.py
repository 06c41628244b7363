"""Estimates that keep few windows per shift, or all of very many, enumerate their own: riding along
costs by the shift and by the window, whatever they keep.  Each result equals the query run alone."""
import pytest

from paper_1810_00980_gb300 import synth

pytestmark = pytest.mark.gpu

KEYS = ("status", "count", "estimate", "windows", "windows_kept", "var_hat", "shift_var", "p_used")


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    small = tm.Graph(*(torch.from_numpy(x).cuda() for x in synth.chung_lu_hawkes(700, 40_000, 2.1, seed=13, horizon=2_000_000)), 700)
    large = tm.Graph(*synth.chung_lu_hawkes_gpu(10_000, 1_000_003, 2.1, 4), 10_000)
    yield tm, small, large
    small.free()
    large.free()


def _alone(tm, g, q, r):
    one = tm.run_batch(g, [q])[0]
    assert {k: r[k] for k in KEYS} == {k: one[k] for k in KEYS}


@pytest.mark.parametrize("name", ["cycle3", "pingpong", "cycle4"])
def test_many_sparse_seeds_stay_apart(env, name):
    tm, small, _ = env
    mo = tm.Motif(*synth.MOTIFS[name])
    qs = [tm.estimate_query(mo, 3600, 2, 0.001, s) for s in range(2000)]
    res = tm.run_batch(small, qs)
    assert sum(r["first_edges"] > 0 for r in res) > 100      # (those that kept a window with edges)
    for k in range(0, 2000, 97):
        _alone(tm, small, qs[k], res[k])


def test_many_sparse_shifts_do_not_ride_on_an_exact_query(env):
    tm, small, _ = env
    mo = tm.Motif(*synth.MOTIFS["cycle3"])
    qs = [tm.exact_query(mo, 3600), tm.estimate_query(mo, 3600, 10, 1e-4, 3, b=20_000), tm.estimate_query(mo, 3600, 10, 0.9, 4)]
    res = tm.run_batch(small, qs)
    assert res[1]["first_edges"] > 0
    for q, r in zip(qs, res):
        _alone(tm, small, q, r)


@pytest.mark.parametrize("name", ["cycle3", "pingpong"])
def test_every_window_of_very_many_stays_one_slot(env, name):
    tm, small, _ = env
    mo = tm.Motif(*synth.MOTIFS[name])
    qs = [tm.estimate_query(mo, 1, 10, 1.0, 1), tm.estimate_query(mo, 10, 1, 1.0, 2), tm.estimate_query(mo, 60, 2, 1.0, 3)]
    res = tm.run_batch(small, qs)
    assert all(r["first_edges"] == 40_000 for r in res)
    res = tm.run_batch(small, [tm.exact_query(mo, 3600)] + qs)[1:]
    assert all(r["first_edges"] == 40_000 for r in res)
    for q, r in zip(qs, res):
        _alone(tm, small, q, r)


def test_dense_and_sparse_seeds_of_one_motif(env):
    tm, _, large = env
    mo = tm.Motif(*synth.MOTIFS["cycle3"])
    dense = [tm.estimate_query(mo, 3600, 10, 0.1, s) for s in range(40)]
    sparse = [tm.estimate_query(mo, 3600, 10, 0.0005, 100 + s) for s in range(400)]
    res = tm.run_batch(large, dense + sparse)
    assert sum(r["first_edges"] > 0 for r in res[:40]) == 1  # one enumeration for the dense ones
    assert sum(r["first_edges"] > 0 for r in res[40:]) > 40
    for k in (0, 17, 39, 41, 200, 439):
        _alone(tm, large, (dense + sparse)[k], res[k])
