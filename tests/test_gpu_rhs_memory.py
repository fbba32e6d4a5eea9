"""bssn_rhs of a caller's register writes nothing but its output: a float64 or
double-word context's own memory (state, stage buffers, anchors, geometry
table) holds the same bytes before and after, in every form of the stage (tiles
with and without groups of threads; one point at a time for a register that is
not 16-byte aligned), so that captured calls may run beside one another and
beside the context's steps."""
import numpy as np
import pytest

import cases as T
import oracle as O
from paper_1111_3344_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(16, 12, 9), (74, 21, 36)])
@pytest.mark.parametrize("boundary", ["sommerfeld", "periodic"])
@pytest.mark.parametrize("precision", ["fp64", "ff"])
@pytest.mark.parametrize("odd", [False, True])
def test_context_memory_is_untouched(n, boundary, precision, odd):
    import torch
    from paper_1111_3344_gb300 import bssn as B
    c = dict(n=n, xmin=(-0.9, -1.1, -0.7), h=0.11, boundary=boundary, precision=precision)
    st = inputs.random_state(3, n, c["xmin"], c["h"], amp=0.05)
    if boundary == "periodic":
        st = O.fill_periodic(T.oracle_cfg(c), st)
    evo = B.Evolution(T.gpu_params(c))
    evo.set_state(st)
    evo.rk4_step(1)
    reg = evo.numpy_to_register(st)
    if odd:
        r = torch.empty(reg.numel() + 1, dtype=reg.dtype, device=reg.device)[1:].view(reg.shape)
        reg = r.copy_(reg)
    out = torch.zeros_like(reg)
    torch.cuda.synchronize()
    before = evo.mem.clone()
    B.bssn_rhs(evo.ctx, reg.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(before, evo.mem)
    want, mag = O.rhs_mag(T.oracle_cfg(c), st)
    got = evo.register_to_numpy(out)
    inner = np.s_[:, 3:-3, 3:-3, 3:-3] if boundary == "periodic" else np.s_[:]
    assert T.rounding_aware_errors(got[inner], want[inner], mag[inner]).max() <= 1.0
    evo.close()
