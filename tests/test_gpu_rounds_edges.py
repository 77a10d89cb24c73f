"""GPU parity of the round-based finishes above the 65,536 edges from which they
remember finished edges and sent messages: edge counts off the 32-edge chunks,
hot receivers, long chains (many rounds), forests, and plans whose second
contents keep other edges alive."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu
LINE = 1 << 16


def _graphs():
    for m in (LINE - 1, LINE, LINE + 1, LINE + 31, LINE + 33):
        yield f"m{m}", 20011, graphgen.er(20011, m, m)
    n, e = graphgen.grid_paths(200, 0.05, 4, 20001, 9)                 # chains of 20,001: many rounds
    yield "chains", n, e
    n = 120000                                                         # every edge aims at one of seven receivers
    hubs = np.stack([np.arange(n) % 7 + n - 7, np.arange(n)], 1).astype(np.uint32)
    yield "hubs", n, np.concatenate([hubs, hubs[::-1], graphgen.er(n, 501, 3)])
    low = np.stack([np.arange(n) % 5, np.arange(n)], 1).astype(np.uint32)   # ... and one of five lowest ids
    yield "low_hubs", n, np.concatenate([low, graphgen.er(n, 30001, 4)])


GRAPHS = list(_graphs())
RULES = [("sv", "PRF"), ("lt", "PRF"), ("lt", "PUF"), ("lt", "PRS"), ("lt", "EUS"), ("lt", "CRFA"), ("stergiou", "PRF")]


def test_the_graphs_lie_above_the_line():
    assert all(len(e) > LINE for name, _, e in GRAPHS if name in ("chains", "hubs", "low_hubs"))


@pytest.mark.parametrize("link,lt", RULES)
def test_labels(link, lt):
    g.build()
    v = g.make_variant(link=link, lt=lt)
    for name, n, e in GRAPHS:
        ref = oracle.cc_uf(n, e)
        lab = g.cc(n, dev(e), v)
        off, cols = graphgen.csr(n, e)
        labc = g.cc_csr(n, dev(off), dev(cols), v)
        g.gconn_sync()
        assert (host_u32(lab) == ref).all(), name
        assert (host_u32(labc) == ref).all(), name


@pytest.mark.parametrize("link,lt", [("sv", "PRF"), ("lt", "PRF"), ("lt", "PRS"), ("lt", "CRFA")])
def test_forests(link, lt):
    """Valid; with full compression also the same every time (the smallest (label, edge id) wins)."""
    g.build()
    v = g.make_variant(link=link, lt=lt)
    for name, n, e in GRAPHS:
        ref = oracle.cc_uf(n, e)
        runs = []
        for _ in range(2):
            ids, _ = g.spanning_forest(n, dev(e), v)
            g.gconn_sync()
            runs.append(np.sort(ids.cpu().numpy().astype(np.uint64)))
            assert oracle.sf_check(n, e, runs[-1], ref) == 0, name
        assert lt == "PRS" or (runs[0] == runs[1]).all(), name


@pytest.mark.parametrize("link", ["sv", "lt"])
@pytest.mark.parametrize("csr", [False, True])
def test_plan_replays_on_new_contents(link, csr):
    """The second contents are the first with every second 4,096-edge piece made of repeats of one edge (and
    the rows of the CSR permuted), so that other chunks finish early; then the first again."""
    import torch
    n, m = 50000, 100003
    e1 = graphgen.er(n, m, 1)
    e2 = graphgen.er(n, m, 2)
    for k in range(0, m, 8192):
        e2[k:k + 4096] = e2[0]
    v = g.make_variant(link=link)
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    if csr:
        (o1, c1), (o2, c2) = graphgen.csr(n, e1), graphgen.csr(n, e2)
        size = max(len(c1), len(c2))
        off, cols = dev(o1 if len(c1) == size else o2), torch.zeros(size, dtype=torch.int32, device="cuda")
        p = g.gconn_plan_create_cc_csr(n, off, cols, lab, v)       # the plan's lists are sized for the larger one
        pairs = ((o1, c1, e1), (o2, c2, e2), (o1, c1, e1))
    else:
        d = dev(e1)
        p = g.gconn_plan_create_cc(n, m, d, lab, v)
        pairs = ((None, None, e1), (None, None, e2), (None, None, e1))
    for o, c, e in pairs:
        if csr:
            off.copy_(dev(o))
            cols[:len(c)].copy_(dev(c))
        else:
            d.copy_(dev(e))
        g.gconn_plan_run(p)
        g.gconn_sync()
        assert (host_u32(lab) == oracle.cc_uf(n, e)).all()
    g.gconn_plan_destroy(p)
