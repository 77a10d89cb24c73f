"""GPU parity of HB sampling under the rules without on-the-fly compression on
both sides of the vertex count where its second step climbs longer before it
defers a union."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 19) - 1, 1 << 19, (1 << 19) + 33])
@pytest.mark.parametrize("link", ["async", "hooks", "afforest"])
def test_labels(n, link):
    """A third of the vertices on permuted paths (long walks), the rest uniform random."""
    g.build()
    k = n // 3
    p = graphgen.permutation(k, n)
    e = np.concatenate([np.stack([p[:-1], p[1:]], 1), graphgen.er(n - k, n, 3) + np.uint32(k)]).astype(np.uint32)
    off, cols = graphgen.csr(n, e)
    lab = g.cc_csr(n, dev(off), dev(cols), g.make_variant(sample="hb", link=link))
    g.gconn_sync()
    assert (host_u32(lab) == oracle.cc_uf(n, e)).all()
