"""A wait between tiles that expires ends the call with TM_ECUDA, and nothing behind it uses what the
waiting kernel did not write.  The bounds-checked build leaves the first tile of one launch to
nobody (tm_check_expire), launch after launch: the sort passes of the graph build, the partition by
windows, the scans of the windows and of the range lengths, in a batch, a captured batch and the
count without allocation.  No bounds check may fire, and the same calls work right afterwards."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
from paper_1810_00980_gb300 import synth, tm
assert tm.LIB_PATH.endswith("libtmotif_checked.so"), tm.LIB_PATH
torch.cuda.set_device(0)
assert tm.check_status(clear=True) == 0
cycle3, outstar3, path2 = tm.Motif([0, 1, 2], [1, 2, 0]), tm.Motif([2, 2, 2], [0, 1, 0]), tm.Motif([0, 1], [1, 2])

def queries(d):
    # partitioned by windows; more windows than a scan tile; exact counts
    return [tm.estimate_query(cycle3, 40_000 * d, 5, 0.5, 3), tm.estimate_query(path2, 10 * d, 2, 0.1, 4),
            tm.exact_query(outstar3, 3_600 * d)]

def status(f):
    try:
        return 0, f()
    except tm.TmError as e:
        return e.status, None

def same(a, b):
    return [(r["status"], r["count"], r["estimate"]) for r in a] == [(r["status"], r["count"], r["estimate"]) for r in b]

def each_launch(f, ok):
    "f with its 1st, 2nd, ... waiting launch expiring, until there is none left; how many there were"
    for nth in range(1, 100):
        assert tm.check_expire(nth) == 0
        s, r = status(f)
        if tm.check_expire(0):
            assert s == 0 and ok(r)
            return nth - 1
        torch.cuda.synchronize()
        word = tm.check_status(clear=True)
        assert s == tm.TM_ECUDA and word == 0, (nth, s, hex(word))
        s, r = status(f)
        assert s == 0 and ok(r), (nth, s)

src, dst, t = synth.chung_lu_hawkes(1500, 60_000, 2.1, seed=9, horizon=2_000_000)
for ticks in (1, 1 << 20):   # 32-bit and 64-bit times
    edges = tuple(torch.from_numpy(x).cuda() for x in (src, dst, t * ticks))
    qs = queries(ticks)
    with tm.Graph(*edges, 1500) as g:
        want = tm.run_batch(g, qs)
        assert all(r["count"] > 0 for r in want)
        n = each_launch(lambda: tm.run_batch(g, qs), lambda r: same(r, want))
        assert n >= 3, n
        def captured():
            pb = tm.PreparedBatch(g, qs)
            try:
                pb.launch()
                return pb.results()
            finally:
                pb.free()
        assert each_launch(captured, lambda r: same(r, want)) == 2
        def noalloc():
            out = ctypes.c_int64(-1)
            s = tm.lib().tm_count_exact_noalloc(g.handle, outstar3.handle, 3_600 * ticks, None, ctypes.byref(out))
            if s:
                raise tm.TmError(s, "noalloc")
            return out.value
        assert each_launch(noalloc, lambda r: r == want[2]["count"]) == 1
    def build():
        with tm.Graph(*edges, 1500) as h:
            return tm.run_batch(h, qs[2:])
    n = each_launch(build, lambda r: same(r, want[2:]))
    assert n >= 5, n   # two passes of two sorts, the range lengths

# more first edges than one scan launch takes, behind a partition that was not finished
m, n = 1_100_003, 5_000
s, d, t = synth.chung_lu_hawkes_gpu(n, m, 2.1, 3)
with tm.Graph(s, d, t, n) as g:
    qs = [tm.estimate_query(cycle3, 86_400, 30, 0.5, 3), tm.exact_query(outstar3, 3_600), tm.exact_query(path2, 60),
          tm.exact_query(tm.Motif([0, 1], [1, 0]), 60)]
    want = tm.run_batch(g, qs)
    assert each_launch(lambda: tm.run_batch(g, qs), lambda r: same(r, want)) >= 1
print("expired ok")
"""


def test_expired_waits_end_with_an_error_and_leave_nothing_behind():
    import __graft_entry__
    __graft_entry__.build()
    env = dict(os.environ, TMOTIF_CHECKED="1")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "expired ok" in r.stdout, (r.stdout[-2000:], r.stderr[-4000:])


def test_ordinary_build_refuses():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    if tm.LIB_PATH.endswith("libtmotif_checked.so"):
        pytest.skip("this process loaded the checked build")
    with pytest.raises(tm.TmError) as e:
        tm.check_expire(1)
    assert e.value.status == tm.TM_EINVAL
