"""The bounded waits of the float64 stage in tiles (csrc/k_stage_fx.cu) where they
run out, without a GPU fault: test hooks leave a copy out and let its wait give
up after a few polls, with nothing else in flight.  Every group of threads at
once, or one copy among the many that a tile loads one after another: the first,
a middle and the last round, before and after the groups part.  Checked: the
timeout is reported once, no interior point of the result is written, and with
the hook off the context (or batch) gives the bits of a fresh one."""
import numpy as np
import pytest

import cases as T
from paper_1111_3344_gb300 import inputs

pytestmark = pytest.mark.gpu

ETIMEOUT = 5
GROUPS4, ONE = (24, 20, 18), (74, 21, 36)  # 75 tiles, in four groups of threads; 540 tiles
AT = [(GROUPS4, None)] + [(GROUPS4, (g, r)) for g, r in ((0, 0), (0, 2), (1, 0), (2, 1), (3, 2), (1, 3), (2, 4), (3, 6))]
AT += [(ONE, None)] + [(ONE, (0, r)) for r in (0, 1, 8, 10, 23)]


def _case(n, precision="fp64", boundary="sommerfeld"):
    return dict(n=n, xmin=(-0.9, -1.1, -0.7), h=0.11, boundary=boundary, precision=precision)


def _state(c):
    return inputs.random_state(13, c["n"], c["xmin"], c["h"], amp=0.03)


@pytest.mark.parametrize("n,at", AT)
@pytest.mark.parametrize("precision", ["fp64", "ff"])
def test_wait_timeout_is_reported_and_recovered(n, at, precision):
    import torch
    from paper_1111_3344_gb300 import bssn as B
    c = _case(n, precision)
    st = _state(c)
    ref = B.Evolution(T.gpu_params(c))
    ref.set_state(st, 0.0)
    ref.rk4_step(1)
    want, _ = ref.get_state()
    ref.close()

    def stall(polls):
        if at is None or polls == 0:
            B.bssn_test_stall_tma(evo.ctx, polls)
        else:
            B.bssn_test_stall_tile(evo.ctx, polls, *at)

    evo = B.Evolution(T.gpu_params(c))
    evo.set_state(st, 0.0)
    stall(64)
    evo.rk4_step(1)
    with pytest.raises(B.BssnError) as e:
        B.bssn_wait_state(evo.ctx)
    assert e.value.status == ETIMEOUT
    B.bssn_wait_state(evo.ctx)  # the error word was cleared when read
    reg = evo.numpy_to_register(st)
    out = torch.full_like(reg, 7.0)
    torch.cuda.synchronize()
    B.bssn_rhs(evo.ctx, reg.data_ptr(), out.data_ptr())
    with pytest.raises(B.BssnError) as e:
        B.bssn_wait_state(evo.ctx)
    assert e.value.status == ETIMEOUT
    assert (evo.register_to_numpy(out)[:, 3:-3, 3:-3, 3:-3] == 7.0).all()
    stall(0)
    evo.set_state(st, 0.0)
    evo.rk4_step(1)
    got, _ = evo.get_state()
    assert np.array_equal(got, want)
    evo.close()


@pytest.mark.parametrize("precision", ["fp64", "ff"])
def test_batch_wait_timeout_is_reported_and_recovered(precision):
    from paper_1111_3344_gb300 import bssn as B
    cases = [_case(GROUPS4, precision), _case(ONE, precision, "periodic")]
    states = [_state(c) for c in cases]
    params = [T.gpu_params(c) for c in cases]

    def make():
        b = B.Batch(precision, pool_bytes=sum(B.Batch.member_bytes(p) for p in params) + (16 << 20), max_members=4)
        ids = [b.add(p) for p in params]
        return b, ids

    def run(b, ids):
        for i, s in zip(ids, states):
            b.set_state(i, s, 0.0)
        b.step(1)

    ref, ids = make()
    run(ref, ids)
    want = [ref.get_state(i)[0] for i in ids]
    ref.close()
    b, ids = make()
    B.bssn_batch_test_stall_tma(b.handle, 64)
    run(b, ids)
    with pytest.raises(B.BssnError) as e:
        b.get_state(ids[0])
    assert e.value.status == ETIMEOUT
    b.get_state(ids[0])  # cleared when read
    B.bssn_batch_test_stall_tma(b.handle, 0)
    run(b, ids)
    for i, w in zip(ids, want):
        assert np.array_equal(b.get_state(i)[0], w)
    b.close()


def test_stalled_copy_is_in_range():
    from paper_1111_3344_gb300 import bssn as B
    evo = B.Evolution(T.gpu_params(_case((8, 8, 8))))
    for polls, group, rd in ((-1, 0, 0), ((1 << 20) + 1, 0, 0), (1, -1, 0), (1, 4, 0), (1, 0, -1), (1, 0, 24)):
        with pytest.raises(B.BssnError):
            B.bssn_test_stall_tile(evo.ctx, polls, group, rd)
    evo.close()
