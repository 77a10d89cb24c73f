"""GPU parity of the batched kernel at the edges of its edge groups (8 x 32
edges per warp turn), of its 16-bit id pairs and of its shared-memory layouts."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


def _batch(graphs):
    vo = np.cumsum([0] + [n for n, _ in graphs]).astype(np.uint64)
    eo = np.cumsum([0] + [len(e) for _, e in graphs]).astype(np.uint64)
    return vo, eo, np.concatenate([e for _, e in graphs]).astype(np.uint32)


def _path(n, seed):
    p = graphgen.permutation(n, seed)
    return np.stack([p[:-1], p[1:]], 1)


CASES = {
    # edge counts around the lane, row, group and block strides
    "edge_counts": [(97, graphgen.er(97, m, 10 + m)) for m in
                    (0, 1, 31, 32, 33, 255, 256, 257, 2047, 2048, 2049, 8191, 8192, 8193)],
    # the largest ids, both layouts of the parents and their limit
    "id_limits": [(n, graphgen.er(n, n + 5, n)) for n in (1, 2, 33, 52975, 52976, 52977, 58112, 65535, 65536)],
    # long climbs: permuted and reversed paths, a star at its largest id
    "climbs": [(65536, _path(65536, 3)), (50001, _path(50001, 4)),
               (40000, np.stack([np.arange(39999, 0, -1), np.arange(39998, -1, -1)], 1)),
               (4097, np.stack([np.full(4096, 4096), np.arange(4096)], 1))],
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("rule", [("async", "halve"), ("remcas", "naive")])
@pytest.mark.parametrize("block", [32, 1024])
def test_matches_oracle(name, rule, block):
    import torch
    g.build()
    vo, eo, e = _batch(CASES[name])
    t = g.gconn_batch_tune_default()
    for c in range(g.GCONN_BATCH_CLASSES):
        t.block[c], t.link[c], t.find[c] = block, g.LINKS[rule[0]], g.FINDS[rule[1]]
    lab = torch.empty(int(vo[-1]), dtype=torch.int32, device="cuda")
    g.gconn_cc_batched(len(vo) - 1, vo, eo, dev(e), lab, t)
    g.gconn_sync()
    assert (host_u32(lab) == oracle.batched_cc(vo, eo, e)).all()


def test_range_error_is_reported_and_the_rest_is_exact():
    import torch
    g.build()
    vo, eo, e = _batch([(500, graphgen.er(500, 900, 1)), (300, graphgen.er(300, 500, 2))])
    ref = oracle.batched_cc(vo, eo, e)
    e[901, 1] = 300                       # one edge of the second graph leaves it
    lab = torch.empty(int(vo[-1]), dtype=torch.int32, device="cuda")
    g.gconn_cc_batched(2, vo, eo, dev(e), lab, None)
    with pytest.raises(g.GconnError) as x:
        g.gconn_sync()
    assert x.value.status == g.GCONN_E_RANGE
    assert (host_u32(lab)[:500] == ref[:500]).all()
