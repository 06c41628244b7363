"""The bounds-checked build on graphs of more than 2^21 edges: the pair table is filled part by
part (and, when every pair hashes into one list, in one part after all), the range lengths are
scanned by more tiles than one launch takes, and the matcher's chunks start from the noted items.
Counts of two-edge motifs against numpy, and no check may fire."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
from paper_1810_00980_gb300 import tm
assert tm.LIB_PATH.endswith("libtmotif_checked.so"), tm.LIB_PATH
torch.cuda.set_device(0)
assert tm.check_status(clear=True) == 0
rng = np.random.default_rng(8)
n, m, delta, span = 20_000, (3 << 20) + 1, 20_000, 100_000
u, v = rng.integers(0, n, 6_000_000), rng.integers(0, n, 6_000_000)
for crowded in (False, True):
    if crowded:   # pairs of one list only (SplitMix64 of the pair, its upper six bits)
        x = (u.astype(np.uint64) << np.uint64(32)) | v.astype(np.uint64)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        keep = np.flatnonzero(((x ^ (x >> np.uint64(31))) >> np.uint64(58)) == 5)
        pick = keep[rng.integers(0, len(keep), m)]
        src, dst = u[pick].astype(np.int32), v[pick].astype(np.int32)
    else:
        h = m // 2   # replies are common
        src = np.concatenate([u[:h], v[:m - h]]).astype(np.int32)
        dst = np.concatenate([v[:h], u[:m - h]]).astype(np.int32)
        order = rng.permutation(m)
        src, dst = src[order], dst[order]
    t = np.sort(rng.integers(0, 50_000, m)).astype(np.int64)
    own = (src.astype(np.int64) * n + dst) * span + t
    rev = (dst.astype(np.int64) * n + src) * span + t
    keys, ok = np.sort(own), src != dst
    after = lambda k: int((np.searchsorted(keys, k + delta, "right") - np.searchsorted(keys, k, "right"))[ok].sum())
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), n) as g:
        assert g.info().n_pairs == len(np.unique(own // span))
        r = tm.run_batch(g, [tm.exact_query(tm.Motif([0, 1], [1, 0]), delta), tm.exact_query(tm.Motif([0, 0], [1, 1]), delta)])
        assert [x["count"] for x in r] == [after(rev), after(own)], crowded
    torch.cuda.synchronize()
    word = tm.check_status(clear=True)
    assert word == 0, f"bounds checks fired: {word:#x}"
print("checked ok")
"""


def test_checked_build_runs_clean_beyond_2_to_21_edges():
    import __graft_entry__
    __graft_entry__.build()
    env = dict(os.environ, TMOTIF_CHECKED="1")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "checked ok" in r.stdout, (r.stdout[-2000:], r.stderr[-4000:])
