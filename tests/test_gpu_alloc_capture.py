"""A context made while the calling thread captures another stream: making it
calls nothing that a capture refuses, so that neither the capture nor the
context is lost.  Both run afterwards."""
import numpy as np
import pytest

import cases as T
from paper_1111_3344_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "ff"])
@pytest.mark.parametrize("boundary", ["sommerfeld", "periodic"])
def test_context_made_during_a_capture(precision, boundary):
    import torch
    from paper_1111_3344_gb300 import bssn as B
    c = dict(n=(16, 12, 9), xmin=(-0.9, -1.1, -0.7), h=0.11, boundary=boundary, precision=precision)
    st = inputs.random_state(3, c["n"], c["xmin"], c["h"], amp=0.05)
    evo = B.Evolution(T.gpu_params(c))  # (and the kernels are loaded)
    evo.set_state(st)
    evo.rk4_step(2)
    want = evo.get_state()[0]
    p = T.gpu_params(c)
    nbytes = B.bssn_required_bytes(p)
    mem = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    own, other = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=other):
        x.add_(1.0)
        ctx = B.bssn_alloc(p, mem.data_ptr(), nbytes, own.cuda_stream)
        x.add_(1.0)
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 2.0).all()
    host = np.ascontiguousarray(st)
    B.bssn_set_state(ctx, host, 0.0)
    B.bssn_rk4_step(ctx, 2)
    out = np.empty_like(host)
    B.bssn_get_state(ctx, out)
    assert np.array_equal(out, want)
    B.bssn_free(ctx)
    evo.close()
