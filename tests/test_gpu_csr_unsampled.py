"""GPU parity of the unsampled CSR finish on graphs large enough for its
compared-and-queued form: long rows cut into tasks, long and short low-degree
lists, the overflow list, forests, 32- and 64-bit offsets."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import UF_COMBOS, UF_FOREST, combo_id, dev, host_u32

pytestmark = pytest.mark.gpu
N = 1 << 18


def _hubs(n):
    """Rows of 1 to 70,001 arcs: hubs in the middle of the ids, the rest of degree 1 to 3."""
    ids = np.arange(n, dtype=np.uint32)
    parts = [np.stack([np.full(k, h), ids[s:s + k]], 1) for h, s, k in
             ((n // 2, 5, 70001), (n // 2 + 1, 100, 257), (n // 2 + 2, 60000, 256), (n // 2 + 3, 7, 33), (9, 0, 512))]
    return np.concatenate(parts + [graphgen.er(n, n // 3, 4)]).astype(np.uint32)


GRAPHS = {"hubs": (N, lambda: _hubs(N)), "sparse_ragged": (N + 77, lambda: graphgen.er(N + 77, N // 2, 5)),
          "rmat": (N, lambda: graphgen.rmat(18, 16 * N + 3, 6)), "few_rows": (N, lambda: _hubs(N)[:70300])}


@pytest.fixture(scope="module")
def built():
    g.build()
    out = {}
    for name, (n, make) in GRAPHS.items():
        e = make()
        off, cols = graphgen.csr(n, e)
        out[name] = (n, off, cols, dev(off), dev(off.astype(np.uint32)), dev(cols), oracle.cc_uf(n, e))
    return out


@pytest.mark.parametrize("combo", UF_COMBOS[::2], ids=combo_id)
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_labels(built, name, combo):
    n, _, _, o64, o32, cols, ref = built[name]
    v = g.make_variant(link=combo[0], find=combo[1], splice=combo[2])
    for off in (o64, o32):
        lab = g.cc_csr(n, off, cols, v)
        g.gconn_sync()
        assert (host_u32(lab) == ref).all()


@pytest.mark.parametrize("combo", UF_FOREST[::4], ids=combo_id)
@pytest.mark.parametrize("name", ["hubs", "rmat"])
def test_forests(built, name, combo):
    n, off, cols, _, o32, dcols, ref = built[name]
    ids, lab = g.spanning_forest_csr(n, o32, dcols, g.make_variant(link=combo[0], find=combo[1], splice=combo[2]),
                                     labels=True)
    g.gconn_sync()
    row = np.repeat(np.arange(n, dtype=np.uint32), np.diff(off).astype(np.int64))
    arcs = np.stack([row, cols], 1)
    assert oracle.sf_check(n, arcs, ids.cpu().numpy().astype(np.uint64), ref) == 0
    assert (host_u32(lab) == ref).all()


def test_overflow_list():
    """More 256-arc tasks than the task array holds: the rest of the rows go one warp a row."""
    g.build()
    e = graphgen.er(N, 40_000_000, 8)
    e[: N // 2] = np.stack([np.arange(N // 2), np.arange(N // 2) + 1], 1)
    off, cols = graphgen.csr(N, e)
    deg = np.diff(off)
    assert ((deg + 255) // 256).sum() > N + 1024
    lab = g.cc_csr(N, dev(off), dev(cols), g.make_variant(link="remcas", splice="split_one"))
    g.gconn_sync()
    assert (host_u32(lab) == oracle.cc_uf(N, e)).all()


def test_out_of_range_column(built):
    n, off, cols, _, o32, _, ref = built["hubs"]
    bad = cols.copy()
    bad[int(off[n // 2]) + 40000] = n          # inside a hub's row
    lab = g.cc_csr(n, o32, dev(bad), g.make_variant(link="remcas", splice="split_one"))
    with pytest.raises(g.GconnError) as x:
        g.gconn_sync()
    assert x.value.status == g.GCONN_E_RANGE
