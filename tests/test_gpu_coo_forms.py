"""GPU parity of the COO finish at the sizes where its forms meet: one block,
a union per thread, a first pass over a sample, one filtered pass."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import UF_COMBOS, UF_FOREST, combo_id, dev, host_u32

pytestmark = pytest.mark.gpu

SIZES = [(16384, 40001), (16385, 40001), (16384, 65536), (16384, 65537), (1, 65536), (2, 3),       # one block
         (9001, 49151), (9001, 49152), (32767, 65535), (32768, 65535), (32768, 65536),             # union per thread
         (1 << 19, 1 << 20), ((1 << 19) + 1, 1 << 20), (40000, 160031), (40000, 159999), (33000, 999999)]


def _graph(n, m):
    """Edges sorted by endpoint for every second size: an ordered list is sampled evenly too."""
    e = graphgen.er(n, m, n + m)
    return e[np.lexsort((e[:, 1], e[:, 0]))] if (n + m) % 2 else e


@pytest.fixture(scope="module")
def graphs():
    g.build()
    out = []
    for n, m in SIZES:
        e = _graph(n, m)
        out.append((n, m, e, dev(e), oracle.cc_uf(n, e)))
    side = np.arange(300 * 300, dtype=np.uint32).reshape(300, 300)      # a long, sorted list of low degree
    e = np.concatenate([np.stack([side[:, :-1].ravel(), side[:, 1:].ravel()], 1),
                        np.stack([side[:-1].ravel(), side[1:].ravel()], 1)])
    out.append((90000, len(e), e, dev(e), oracle.cc_uf(90000, e)))
    return out


@pytest.mark.parametrize("combo", UF_COMBOS, ids=combo_id)
def test_labels(graphs, combo):
    v = g.make_variant(link=combo[0], find=combo[1], splice=combo[2])
    for n, m, e, d, ref in graphs:
        lab = g.cc(n, d, v)
        g.gconn_sync()
        assert (host_u32(lab) == ref).all(), (n, m)


@pytest.mark.parametrize("combo", UF_FOREST[::3], ids=combo_id)
def test_forests(graphs, combo):
    v = g.make_variant(link=combo[0], find=combo[1], splice=combo[2])
    for n, m, e, d, ref in graphs[9:]:
        ids, lab = g.spanning_forest(n, d, v, labels=True)
        g.gconn_sync()
        assert oracle.sf_check(n, e, ids.cpu().numpy().astype(np.uint64), ref) == 0, (n, m)
        assert (host_u32(lab) == ref).all(), (n, m)


@pytest.mark.parametrize("n,m", [(5000, 9000), (9001, 49200), (40000, 200000), (700000, 800000)])
def test_out_of_range_edge_is_reported_and_skipped(n, m):
    """The bad edge is left out; every other edge still counts."""
    g.build()
    e = graphgen.er(n, m, 7)
    bad = e.copy()
    bad[m // 2] = (3, n)
    keep = np.delete(e, m // 2, 0)
    lab = g.cc(n, dev(bad))
    with pytest.raises(g.GconnError) as x:
        g.gconn_sync()
    assert x.value.status == g.GCONN_E_RANGE
    assert (host_u32(lab) == oracle.cc_uf(n, keep)).all()


def test_small_graph_in_a_plan_sees_new_contents():
    import torch
    n, m = 3000, 5000
    e1, e2 = graphgen.er(n, m, 1), graphgen.er(n, m, 2)
    d, lab = dev(e1), torch.empty(n, dtype=torch.int32, device="cuda")
    p = g.gconn_plan_create_cc(n, m, d, lab, g.make_variant(link="async", find="halve"))
    for e in (e1, e2):
        d.copy_(dev(e))
        g.gconn_plan_run(p)
        g.gconn_sync()
        assert (host_u32(lab) == oracle.cc_uf(n, e)).all()
    g.gconn_plan_destroy(p)
