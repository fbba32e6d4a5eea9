"""The autotuners of double-word contexts and batches: the configuration names
that stand for one and the same kernel get one measurement, so that no noise
picks among them, and every name can still be selected."""
import pytest

import cases as T

pytestmark = pytest.mark.gpu

CASE = dict(n=(24, 20, 16), xmin=(-0.9, -1.1, -0.7), h=0.11, boundary="sommerfeld", precision="ff")


def test_context_measures_its_kernel_once():
    from paper_1111_3344_gb300 import bssn as B
    evo = B.Evolution(T.gpu_params(CASE))
    evo.set_initial_data("flat")
    best, ms = B.bssn_autotune(evo.ctx, reps=1)
    names = [B.bssn_tile_name(c) for c in range(B.bssn_tile_count())]
    ff = [c for c, n in enumerate(names) if n.startswith("ff")]
    assert best == ff[0] and len({ms[names[c]] for c in ff}) == 1 and 0.0 < ms[names[ff[0]]] < 1e3
    for c in ff:
        B.bssn_set_tile(evo.ctx, c)
    evo.close()


def test_batch_measures_members_once():
    from paper_1111_3344_gb300 import bssn as B
    p = T.gpu_params(CASE)
    b = B.Batch("ff", pool_bytes=B.Batch.member_bytes(p) + (16 << 20), max_members=2)
    b.set_initial_data(b.add(p), "flat", [])
    best, ms = b.autotune(reps=1)
    names = list(ms)
    ff = [c for c, n in enumerate(names) if n.startswith("ff")]
    assert names[best].startswith("members")
    assert all(ms[names[c]] == ms["members"] > 0.0 for c in ff)
    for c in ff:
        b.set_tile(c)
    b.close()
