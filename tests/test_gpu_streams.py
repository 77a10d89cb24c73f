"""The default stream argument is torch's current stream, also inside a stream
context and after the current device's stream changed."""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2008_11839_gb300 as g
from gpu_util import dev, host_u32

pytestmark = pytest.mark.gpu


def test_handle_follows_the_current_stream():
    import torch
    g.build()
    torch.cuda.init()
    assert g.stream_handle() == (torch.cuda.current_stream().cuda_stream or None)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert g.stream_handle() == s.cuda_stream
        n, e = 3000, graphgen.er(3000, 5000, 1)
        lab = g.cc(n, dev(e))
    assert g.stream_handle() == (torch.cuda.current_stream().cuda_stream or None)
    s.synchronize()
    assert (host_u32(lab) == oracle.cc_uf(n, e)).all()
    assert g.stream_handle(s) == s.cuda_stream and g.stream_handle(0) is None
