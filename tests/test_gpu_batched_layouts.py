"""GPU parity of the batched kernel's two layouts of the parents (32-bit where a
class's largest graph and the warps' queues fit a block's shared memory, 16-bit
above) at their limit, each in a batch of its own, and of small calls and batches
from several threads at once."""
import threading

import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


def _ends(n, seed):
    """A permuted path over all ids (long climbs), edges at the highest ids, random ones."""
    p = graphgen.permutation(n, seed)
    top = np.stack([np.full(64, n - 1), np.arange(n - 65, n - 1)], 1)
    return np.concatenate([np.stack([p[:-1], p[1:]], 1), top, graphgen.er(n, 3 * n, seed)]).astype(np.uint32)


@pytest.mark.parametrize("rule", [("async", "halve"), ("async", "naive"), ("remcas", "naive")])
@pytest.mark.parametrize("block,n", [(1024, 52976), (1024, 52977), (32, 57936), (32, 57937), (1024, 65536), (32, 65536),
                                     (1024, 16385)])
def test_layout_limits(block, n, rule):
    """20 bytes of queue a thread: 52,976 vertices are the last that fit as 32-bit parents with 1,024 threads, 57,936
    with 32.  The second graph is short, so that its edges per thread stay few."""
    import torch
    g.build()
    graphs = [(n, _ends(n, n)), (n - 1, graphgen.er(n - 1, 700, 3))]
    vo = np.cumsum([0] + [k for k, _ in graphs]).astype(np.uint64)
    eo = np.cumsum([0] + [len(e) for _, e in graphs]).astype(np.uint64)
    e = np.concatenate([e for _, e in graphs])
    t = g.gconn_batch_tune_default()
    for c in range(g.GCONN_BATCH_CLASSES):
        t.block[c], t.link[c], t.find[c] = block, g.LINKS[rule[0]], g.FINDS[rule[1]]
    lab = torch.empty(int(vo[-1]), dtype=torch.int32, device="cuda")
    for part in (slice(0, 2), slice(0, 1)):          # together, and the long one alone
        k = part.stop
        g.gconn_cc_batched(k, vo[:k + 1], eo[:k + 1], dev(e), lab, t)
        g.gconn_sync()
        m = int(eo[k])
        assert (host_u32(lab)[:int(vo[k])] == oracle.batched_cc(vo[:k + 1], eo[:k + 1], e[:m])).all()


def test_several_threads_share_the_kernels_limits():
    """Small calls of 10 to 16,384 vertices and batches of different classes from four threads: the kernels'
    shared-memory limit is theirs together, so none may lower it under another."""
    import torch
    g.build()
    cases = []
    for n in (10, 16384, 700, 9001):
        e = graphgen.er(n, 2 * n, n)
        cases.append((n, e, dev(e), oracle.cc_uf(n, e)))
    big = []
    for n in (300, 52976, 4000, 16000):
        e = graphgen.er(n, 2 * n, n)
        big.append((n, e, dev(e), oracle.cc_uf(n, e)))
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                for r in range(30):
                    n, e, d, ref = cases[(k + r) % 4]
                    lab = torch.empty(n, dtype=torch.int32, device="cuda")
                    g.gconn_cc(n, len(e), d, lab, g.make_variant(link="remcas", splice="split_one"))
                    n2, e2, d2, ref2 = big[(k + r) % 4]
                    lab2 = torch.empty(n2, dtype=torch.int32, device="cuda")
                    g.gconn_cc_batched(1, np.array([0, n2], np.uint64), np.array([0, len(e2)], np.uint64), d2, lab2,
                                       None)
                    st.synchronize()
                    assert (host_u32(lab) == ref).all() and (host_u32(lab2) == ref2).all()
        except Exception as x:          # noqa: BLE001 - reported by the main thread
            errors.append(repr(x))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    g.gconn_sync()
    assert not errors, errors[:2]
