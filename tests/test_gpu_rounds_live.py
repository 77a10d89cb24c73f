"""GPU parity of the round-based finishes where edges drop out between rounds:
edge counts off the 32-edge chunks, many rounds, hot receivers, forests, CSR
input and capture."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


def _graphs():
    for m in (1, 31, 32, 33, 63, 64, 65, 4097):
        yield 700, graphgen.er(700, m, m)
    yield graphgen.grid_paths(90, 0.05, 4, 5001, 9)                   # long chains: many rounds
    n = 30000                                                         # every edge aims at a few receivers
    hubs = np.stack([np.arange(n) % 7 + n - 7, np.arange(n)], 1).astype(np.uint32)
    yield n, np.concatenate([hubs, hubs[::-1], graphgen.er(n, 501, 3)])
    yield 1 << 16, graphgen.rmat(16, (1 << 20) + 17, 5)


GRAPHS = list(_graphs())
RULES = [("sv", "PRF"), ("lt", "PRF"), ("lt", "PUF"), ("lt", "PRS"), ("lt", "CRFA"), ("lt", "EUF"), ("stergiou", "PRF")]


@pytest.mark.parametrize("link,lt", RULES)
def test_labels(link, lt):
    g.build()
    v = g.make_variant(link=link, lt=lt)
    for n, e in GRAPHS:
        ref = oracle.cc_uf(n, e)
        lab = g.cc(n, dev(e), v)
        off, cols = graphgen.csr(n, e)
        labc = g.cc_csr(n, dev(off), dev(cols), v)
        g.gconn_sync()
        assert (host_u32(lab) == ref).all(), (n, len(e))
        assert (host_u32(labc) == ref).all(), (n, len(e))


@pytest.mark.parametrize("link,lt", [r for r in RULES if r[1] in ("PRF", "PRS", "CRFA") and r[0] != "stergiou"])
def test_forests(link, lt):
    """Valid; with full compression also the same every time, the winning message being the smallest
    (label, edge id).  (PRS shortens paths in place, so what a jump reads depends on the run.)"""
    g.build()
    v = g.make_variant(link=link, lt=lt)
    for n, e in GRAPHS[7:]:
        runs = []
        for _ in range(2):
            ids, _ = g.spanning_forest(n, dev(e), v)
            g.gconn_sync()
            runs.append(np.sort(ids.cpu().numpy().astype(np.uint64)))
        assert oracle.sf_check(n, e, runs[0], oracle.cc_uf(n, e)) == 0
        assert oracle.sf_check(n, e, runs[1], oracle.cc_uf(n, e)) == 0
        if lt != "PRS":
            assert (runs[0] == runs[1]).all()


@pytest.mark.parametrize("link", ["sv", "lt"])
def test_plan_replays_on_new_contents(link):
    import torch
    n, m = 5000, 20011
    e1, e2 = graphgen.er(n, m, 1), graphgen.er(n, m, 2)
    e2[m // 2:] = e2[0]                       # a sparser second graph: other edges live on
    d, lab = dev(e1), torch.empty(n, dtype=torch.int32, device="cuda")
    p = g.gconn_plan_create_cc(n, m, d, lab, g.make_variant(link=link))
    for e in (e1, e2, e1):
        d.copy_(dev(e))
        g.gconn_plan_run(p)
        g.gconn_sync()
        assert (host_u32(lab) == oracle.cc_uf(n, e)).all()
    g.gconn_plan_destroy(p)
