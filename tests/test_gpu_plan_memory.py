"""A captured round-based pass takes no more device memory than its labels, its
messages and its control words: what only saves time is not a node of a plan,
which a program may hold where memory is short."""
import ctypes

import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu
USED_HIGH = 1   # CU_GRAPH_MEM_ATTR_USED_MEM_HIGH


def _graph_memory(reset=False):
    cu = ctypes.CDLL("libcuda.so.1")
    d, x = ctypes.c_int(), ctypes.c_uint64(0)
    assert cu.cuDeviceGet(ctypes.byref(d), 0) == 0
    f = cu.cuDeviceSetGraphMemAttribute if reset else cu.cuDeviceGetGraphMemAttribute
    assert f(d, USED_HIGH, ctypes.byref(x)) == 0
    return x.value


@pytest.mark.parametrize("link", ["sv", "lt"])
def test_scratch_of_a_captured_pass_does_not_grow_with_the_edges(link):
    """n = 1,000 needs some 12 KB, counted in pages of 32 MiB; one bit per edge of m = 2^29 would be 64 MiB."""
    import torch
    g.build()
    n, m = 1000, 1 << 29
    e = graphgen.er(n, 1 << 16, 3)
    d = dev(e).repeat(m // len(e), 1)
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    p = g.gconn_plan_create_cc(n, m, d, lab, g.make_variant(link=link))
    _graph_memory(reset=True)
    g.gconn_plan_run(p)
    g.gconn_sync()
    used = _graph_memory()
    g.gconn_plan_destroy(p)
    assert (host_u32(lab) == oracle.cc_uf(n, e)).all()
    assert 0 < used < 64 << 20, used
