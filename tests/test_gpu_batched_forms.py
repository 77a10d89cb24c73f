"""GPU parity of the batched kernel's forms (a union per thread, two rows and
eight rows of edges a turn) where they meet: mean edge counts around 4 and 64
a thread, graphs of fewer edges than a warp, a block or a turn."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


def _run(graphs, block, rule):
    import torch
    vo = np.cumsum([0] + [n for n, _ in graphs]).astype(np.uint64)
    eo = np.cumsum([0] + [len(e) for _, e in graphs]).astype(np.uint64)
    e = np.concatenate([e for _, e in graphs]).astype(np.uint32)
    t = g.gconn_batch_tune_default()
    for c in range(g.GCONN_BATCH_CLASSES):
        t.block[c], t.link[c], t.find[c] = block, g.LINKS[rule[0]], g.FINDS[rule[1]]
    lab = torch.empty(int(vo[-1]), dtype=torch.int32, device="cuda")
    g.gconn_cc_batched(len(graphs), vo, eo, dev(e), lab, t)
    g.gconn_sync()
    assert (host_u32(lab) == oracle.batched_cc(vo, eo, e)).all()


@pytest.mark.parametrize("rule", [("async", "naive"), ("async", "halve"), ("remcas", "naive")])
@pytest.mark.parametrize("block", [32, 64, 256, 1024])
def test_mean_edges_around_the_lines(block, rule):
    """One class: every graph with the same edge count, just below, at and above 1, 4 and 64 a thread, as a few graphs
    and (short lists only) as more graphs than blocks are resident."""
    g.build()
    for per in (1, 4, 64):
        for m in (per * block - 1, per * block, per * block + 33):
            _run([(701 + k, graphgen.er(701 + k, m, m + k)) for k in range(5)], block, rule)
            if m <= 20000 and block > 32:
                base = [(701 + k, graphgen.er(701 + k, m, m + k)) for k in range(3)]
                _run(base * (max(2600 // (block // 32), 200)), block, rule)


@pytest.mark.parametrize("block", [32, 256, 1024])
def test_tiny_and_uneven_graphs(block):
    """Hundreds of graphs of 1 to 40 vertices beside one long list in the same class, and out-of-range edges nowhere."""
    g.build()
    small = [(1 + k % 40, graphgen.er(1 + k % 40, (k * 7) % 90, k)) for k in range(400)]
    for big in (0, 2 * block * 8 + 5, 60000):
        _run(small + [(1000, graphgen.er(1000, big, 9))], block, ("remcas", "naive"))


def test_range_error_in_each_form():
    import torch
    g.build()
    for m in (100, 5000, 40000):                 # 0.4, 20 and 156 edges a thread
        e = graphgen.er(900, m, m)
        e[m // 2] = (5, 900)
        vo, eo = np.array([0, 900], np.uint64), np.array([0, m], np.uint64)
        lab = torch.empty(900, dtype=torch.int32, device="cuda")
        g.gconn_cc_batched(1, vo, eo, dev(e), lab, None)
        with pytest.raises(g.GconnError) as x:
            g.gconn_sync()
        assert x.value.status == g.GCONN_E_RANGE
        assert (host_u32(lab) == oracle.cc_uf(900, np.delete(e, m // 2, 0))).all()
