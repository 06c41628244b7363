"""Many second-edge candidates per first edge (more than the item starts noted for a batch), and
first-edge counts on both sides of the step between small and large item grains: in-edge then
out-edge of one hub, against the closed form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m_in,m_out", [(3_000, 400), (3_000, 65), (530_000, 40), (2_090_000, 5), (2_200_000, 5)])
@pytest.mark.parametrize("prepared", [False, True])
def test_every_in_edge_sees_every_out_edge(m_in, m_out, prepared):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    torch.cuda.set_device(0)
    from paper_1810_00980_gb300 import tm
    m = m_in + m_out
    # a->h at times 0 .. m_in - 1, then h->b: all of them follow every in-edge; b is one of three nodes
    b = (1 + np.arange(m_out) % 3).astype(np.int32)
    src = np.concatenate([4 + np.arange(m_in) % 1000, np.zeros(m_out)]).astype(np.int32)
    dst = np.concatenate([np.zeros(m_in), b]).astype(np.int32)
    t = np.arange(m, dtype=np.int64)
    edge = [[1, 0], [0, 2]]
    delta = 2 * m
    with tm.Graph(*(torch.from_numpy(x).cuda() for x in (src, dst, t)), 1004) as g:
        # read one by one (a high threshold): every in-edge's whole range is items
        old = tm.get_tuning()["enum_threshold"]
        tm.set_tuning(enum_threshold=1 << 30)
        try:
            qs = [tm.exact_query(tm.Motif(*edge), delta), tm.exact_query(tm.Motif(*edge), m_out)]
            if prepared:
                pb = tm.PreparedBatch(g, qs)
                pb.launch()
                res = pb.results()
                pb.free()
            else:
                res = tm.run_batch(g, qs)
        finally:
            tm.set_tuning(enum_threshold=old)
    assert res[0]["count"] == m_in * m_out
    # within m_out ticks: the last in-edges, the one i ticks before the first out-edge sees m_out - i + 1
    assert res[1]["count"] == sum(m_out - i + 1 for i in range(1, min(m_out, m_in) + 1))
