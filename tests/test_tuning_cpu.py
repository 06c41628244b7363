"""The tuning that is read is the one that runs, so writing it back changes nothing (no device call)."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
sys.path.insert(0, sys.argv[1])
from paper_1810_00980_gb300 import tm
first = tm.get_tuning()
assert first == {"block_threads": 256, "blocks_per_sm": 6, "chunk_items": 256, "enum_threshold": 48}, first
tm.set_tuning(**first)
assert tm.get_tuning() == first
tm.set_tuning(blocks_per_sm=4)
assert tm.get_tuning() == dict(first, blocks_per_sm=4)
tm.set_tuning(**first)
assert tm.get_tuning() == first
print("ok")
"""


def test_default_tuning_is_the_one_that_runs():
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, (r.stdout, r.stderr[-2000:])
