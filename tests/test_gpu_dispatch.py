"""Which kernels a call launches: the size, rule and memory lines of the
dispatch, on both sides of each line, with the results against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


def kernels_of(call):
    """Names of the kernels that `call` launches."""
    g.gconn_profile_enable(True)
    try:
        g.gconn_profile_sync()
        g.gconn_profile_reset()
        call()
        g.gconn_sync()
        g.gconn_profile_sync()
        return {k for k, v in g.gconn_profile_get().items() if v[0]}
    finally:
        g.gconn_profile_enable(False)


def cc_kernels(n, m, edges, v, ref):
    import torch
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    names = kernels_of(lambda: g.gconn_cc(n, m, edges, lab, v))
    assert (host_u32(lab) == ref).all()
    return names


@pytest.mark.parametrize("rule,n,m,one_block", [
    (("remcas", "naive"), 16384, 65536, True), (("remcas", "naive"), 16384, 65537, False),
    (("remcas", "naive"), 16385, 20000, False),
    (("async", "halve"), 4096, 65536, True), (("async", "halve"), 4097, 9000, False),
    (("async", "naive"), 4096, 1024, True), (("async", "naive"), 4096, 1025, False),
    (("async", "naive"), 4096, 20000, False), (("async", "naive"), 16384, 1000, True)])
def test_one_block_limits_on_device_lists(rule, n, m, one_block):
    g.build()
    e = graphgen.er(n, m, n + m)
    v = g.make_variant(link=rule[0], find=rule[1], splice="split_one" if rule[0] == "remcas" else "none")
    assert ("small_cc" in cc_kernels(n, m, dev(e), v, oracle.cc_uf(n, e))) == one_block


@pytest.mark.parametrize("rule,n,m,one_block", [
    (("remcas", "naive"), 16000, 32768, True), (("remcas", "naive"), 16000, 32769, False),
    (("async", "halve"), 4000, 16384, True), (("async", "halve"), 4000, 16385, False),
    (("async", "naive"), 4000, 1024, True), (("async", "naive"), 4000, 1025, False)])
@pytest.mark.parametrize("pinned", [False, True])
def test_one_block_limits_on_host_lists(rule, n, m, one_block, pinned):
    import torch
    g.build()
    e = graphgen.er(n, m, n + m)
    h = torch.from_numpy(e.view(np.int32)).pin_memory() if pinned else e
    v = g.make_variant(link=rule[0], find=rule[1], splice="split_one" if rule[0] == "remcas" else "none")
    assert ("small_cc" in cc_kernels(n, m, h, v, oracle.cc_uf(n, e))) == one_block


@pytest.mark.parametrize("kw", [dict(block=64), dict(block=256), dict(iter_cap=1 << 20)])
def test_own_block_size_or_cap_keeps_the_global_memory_kernels(kw):
    g.build()
    n, m = 3000, 9000
    e = graphgen.er(n, m, 1)
    ref = oracle.cc_uf(n, e)
    assert "small_cc" in cc_kernels(n, m, dev(e), g.make_variant(link="remcas", splice="split_one"), ref)
    assert "small_cc" not in cc_kernels(n, m, dev(e), g.make_variant(link="remcas", splice="split_one", **kw), ref)


# (rule, n, m, sampled first pass)
COO_LINES = [
    ("remcas", "naive", "split_one", 40000, (1 << 17) - 1, False), ("remcas", "naive", "split_one", 40000, 1 << 17, True),
    ("remcas", "naive", "splice", 70000, 139999, False), ("remcas", "naive", "splice", 70000, 140000, True),
    ("remcas", "naive", "split_one", 9000, 71999, False), ("remcas", "naive", "split_one", 9000, 72000, True),
    ("remcas", "naive", "split_one", (1 << 19) + 1, 1 << 21, False),
    ("remcas", "halve", "halve_one", 40000, (1 << 18) - 1, False), ("remcas", "halve", "halve_one", 40000, 1 << 18, True),
    ("early", "naive", "none", 140000, 279999, False), ("early", "naive", "none", 140000, 280000, True),
    ("early", "naive", "none", 140000, 560000, True), ("early", "split", "none", 140000, 560000, False),
    ("early", "naive", "none", 9000, 143999, False), ("early", "naive", "none", 9000, 144000, True),
    ("async", "naive", "none", 40000, 119999, False), ("async", "naive", "none", 40000, 120000, True),
    ("async", "naive", "none", 1 << 18, (1 << 19) - 1, False), ("async", "naive", "none", 1 << 18, 1 << 19, True),
    ("async", "naive", "none", 600000, 1200000, True), ("async", "naive", "none", 600000, 700000, False),
    ("async", "compress", "none", 33000, 65999, False), ("async", "compress", "none", 33000, 66000, True),
    ("async", "naive", "none", 30000, 400000, False), ("hooks", "naive", "none", 33000, 66000, True),
    ("hooks", "naive", "none", 50000, 80000, False), ("afforest", "naive", "none", 600000, 900000, False),
    ("early", "naive", "none", 600000, 1300000, False), ("early", "naive", "none", 600000, 2400000, False),
    ("remlock", "naive", "split_one", 600000, 1300000, False)]


@pytest.mark.parametrize("link,find,splice,n,m,sampled", COO_LINES)
def test_coo_finish_lines(link, find, splice, n, m, sampled):
    g.build()
    e = graphgen.er(n, m, n + m)
    names = cc_kernels(n, m, dev(e), g.make_variant(link=link, find=find, splice=splice), oracle.cc_uf(n, e))
    assert ("union_coo_sample" in names) == sampled and "union_coo" in names


@pytest.mark.parametrize("n,m", [(40000, 70000), (9000, 60000), (9000, 80000), (300000, 450000), (600000, 500000)])
def test_coo_forests_around_the_lines(n, m):
    g.build()
    e = graphgen.er(n, m, n + m)
    ref = oracle.cc_uf(n, e)
    for link, find, splice in (("remcas", "naive", "split_one"), ("early", "halve", "none"), ("async", "naive", "none")):
        ids, _ = g.spanning_forest(n, dev(e), g.make_variant(link=link, find=find, splice=splice))
        g.gconn_sync()
        assert oracle.sf_check(n, e, ids.cpu().numpy().astype(np.uint64), ref) == 0


def _csr_call(n, off, cols, v, bits):
    import torch
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    f = g.gconn_cc_csr32 if bits == 32 else g.gconn_cc_csr
    f(n, off, cols, lab, v)
    g.gconn_sync()
    return host_u32(lab)


@pytest.mark.parametrize("link", ["remcas", "async", "early", "hooks"])
@pytest.mark.parametrize("n,m", [((1 << 18) - 1, 1 << 21), (1 << 18, 1 << 18), (1 << 18, 1 << 20), (1 << 18, (1 << 21) - 1),
                                 (1 << 18, 1 << 21), (1 << 20, 1 << 18), (1 << 20, (1 << 21) - 1), (1 << 20, 1 << 21)])
def test_unsampled_csr_finish_lines(link, n, m):
    """A direct call between 2^18 and 2^20 vertices, and under Rem and Early with naive finds above, leaves the choice to
    the arc count on the device; a plan and all other calls launch the one kernel.  The labels are the oracle's either
    way, also when a plan's contents turn from a sparse graph to a dense one."""
    import torch
    g.build()
    direct = 1 if n < 1 << 18 or (n >= 1 << 20 and link in ("async", "hooks")) else 2
    e = graphgen.er(n, m, n + m)
    off, cols = graphgen.csr(n, e)
    ref = oracle.cc_uf(n, e)
    v = g.make_variant(link=link, splice="split_one" if link == "remcas" else "none")
    assert (_csr_call(n, dev(off), dev(cols), v, 64) == ref).all()
    assert (_csr_call(n, dev(off.astype(np.uint32)), dev(cols), v, 32) == ref).all()
    d_off, lab = dev(off.astype(np.uint32)), torch.empty(n, dtype=torch.int32, device="cuda")
    d_cols = torch.zeros(max(len(cols), 1 << 22), dtype=torch.int32, device="cuda")
    d_cols[:len(cols)].copy_(dev(cols))
    g.gconn_profile_enable(True)
    try:
        g.gconn_profile_sync()
        g.gconn_profile_reset()
        g.gconn_cc_csr32(n, d_off, d_cols, lab, v)
        g.gconn_profile_sync()
        assert g.gconn_profile_get()["finish"][0] == direct
    finally:
        g.gconn_profile_enable(False)
    p = g.gconn_plan_create_cc_csr32(n, d_off, d_cols, lab, v)
    g.gconn_plan_run(p)
    g.gconn_sync()
    assert (host_u32(lab) == ref).all()
    e2 = graphgen.er(n, 1 << 21 if m < 1 << 20 else 1 << 17, 5)
    o2, c2 = graphgen.csr(n, e2)
    d_off.copy_(dev(o2.astype(np.uint32)))
    d_cols[:len(c2)].copy_(dev(c2))
    g.gconn_plan_run(p)
    g.gconn_sync()
    assert (host_u32(lab) == oracle.cc_uf(n, e2)).all()
    g.gconn_plan_destroy(p)
