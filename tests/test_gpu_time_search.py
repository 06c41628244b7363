"""Counts that hinge on the search by time in long node lists: times evenly spread, in a few
bursts, all equal but the ends, and crowded at either end, at the lengths where the search
changes; against a sliding window in numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _times(kind, m, rng):
    if kind == "even":
        t = rng.integers(0, 10 * m, m)
    elif kind == "bursts":
        t = rng.choice(rng.integers(0, 10**9, 5), m) + rng.integers(0, 60, m)
    elif kind == "flat":
        t = np.full(m, 500)
        t[0], t[-1] = 0, 1_000_000
    elif kind == "front":
        t = (rng.random(m) ** 6 * 1e9).astype(np.int64)
    else:
        t = 10**9 - (rng.random(m) ** 6 * 1e9).astype(np.int64)
    return np.sort(t).astype(np.int64)


@pytest.mark.parametrize("kind", ["even", "bursts", "flat", "front", "back"])
@pytest.mark.parametrize("m", [31, 32, 33, 34, 1_000, 70_001])
def test_in_then_out_of_a_hub(kind, m):
    """a->h then h->b (b a new node): every in-edge of the hub searches its out-list."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    rng = np.random.default_rng(m)
    t = _times(kind, 2 * m, rng)
    out = rng.permutation(np.arange(2 * m) % 2 == 0)
    other = (1 + np.arange(2 * m)).astype(np.int32)          # every edge has a node of its own
    src = np.where(out, 0, other).astype(np.int32)
    dst = np.where(out, other, 0).astype(np.int32)
    to = t[out]
    span = int(t[-1] - t[0])
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), 2 * m + 1) as g:
        for delta in (0, 1, 60, max(1, span // 50), span):
            a = np.searchsorted(to, t[~out], "right")
            b = np.searchsorted(to, t[~out] + delta, "right")
            assert tm.count_exact(g, tm.Motif([1, 0], [0, 2]), delta) == int((b - a).sum()), delta
