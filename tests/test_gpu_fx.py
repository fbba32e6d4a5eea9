"""The float64 right-hand side with integer-summed stencils (csrc/fx.cuh,
csrc/rhs_fx.cuh) where it can go wrong: grids that whole tiles fill and grids
that flat blocks cover, values of very different magnitude inside one stencil,
signed zeros, and stencils outside the integer range (huge, tiny, not finite).

Bar: 1e-12 max(S_f, M_pf) as everywhere (cases.rounding_aware_errors).  A
stencil's alignment error is at most 192 2^-54 of its largest value (1.1e-14),
its rounding 2^-53; the some 400 operations of a field's equation add 4e-14 M,
so the bar holds with a factor of 15 to spare."""
import numpy as np
import pytest

import cases as T
import oracle as O
from paper_1111_3344_gb300 import inputs

pytestmark = pytest.mark.gpu


def _rhs(c, st):
    from paper_1111_3344_gb300.bssn import Evolution
    evo = Evolution(T.gpu_params(c))
    out = evo.register_to_numpy(evo.rhs(evo.numpy_to_register(st)))
    evo.close()
    return out


def _case(n, seed, **kw):
    c = dict(n=n, xmin=(-0.9, -1.1, -0.7), h=0.11, boundary="sommerfeld", **kw)
    return c, inputs.random_state(seed, n, c["xmin"], c["h"], amp=0.05)


SMALL = [7, 8, 10, 13, 14, 16, 19, 20, 22, 23]  # fields that may take any size


@pytest.mark.parametrize("n", [(4, 4, 4), (32, 4, 5), (33, 5, 4), (24, 7, 9), (64, 8, 4), (31, 13, 6)])
@pytest.mark.parametrize("conformal", ["W", "phi"])
def test_wide_range_of_magnitudes(n, conformal):
    """Neighbouring values from 1 down to 1e-25, of both signs, and exact zeros of both signs."""
    c, st = _case(n, 3, conformal=conformal)
    rng = np.random.default_rng(17)
    if conformal == "phi":
        st[0] = -0.5 * np.log(st[0])
    for f in SMALL:
        st[f] = 0.05 * rng.uniform(-1, 1, st[f].shape) * 10.0 ** rng.integers(-25, 1, st[f].shape)
        st[f][rng.random(st[f].shape) < 0.1] = -0.0
    cfg = T.oracle_cfg(c)
    want, mag = O.rhs_mag(cfg, st)
    got = _rhs(c, st)
    assert T.rounding_aware_errors(got, want, mag).max() <= 1.0


@pytest.mark.parametrize("scale", [1e-300, 1e-270, 5e-324, 1e300])
def test_stencils_outside_the_integer_range(scale):
    """B^i and Gt^x of such size: their own right-hand sides by the float64 sums."""
    c, st = _case((12, 9, 8), 5)
    st[21:24] *= scale
    want, mag = O.rhs_mag(T.oracle_cfg(c), st)
    got = _rhs(c, st)
    assert T.rounding_aware_errors(got, want, mag).max() <= 1.0
    if scale < 1.0:  # a stencil of subnormals is not flushed: B's advection is of its size
        st2 = st.copy()
        st2[21:24] = 0.0
        keep = [f for f in range(24) if f not in (21, 22, 23)]
        assert np.abs(got[keep] - _rhs(c, st2)[keep]).max() <= 10 * scale


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("f", [0, 3, 7, 9, 15, 17, 19, 22])
def test_not_finite_values_spread_with_the_stencils(f, bad):
    """One such value: every point whose dissipation stencil holds it is not
    finite in that field, and nothing is where the oracle is finite.  (The
    oracle also multiplies it by the zero coefficients of its stencils, so
    its own set may be larger.)"""
    c, st = _case((16, 9, 8), 7)
    at = (7, 8, 9)
    st[(f,) + at] = bad
    with np.errstate(all="ignore"):
        want = O.rhs(T.oracle_cfg(c), st)
    got = _rhs(c, st)
    inner = np.s_[:, 3:-3, 3:-3, 3:-3]
    assert not (np.isfinite(want[inner]) & ~np.isfinite(got[inner])).any()
    for d in range(3):
        for m in range(-3, 4):
            q = list(at)
            q[d] += m
            if all(3 <= q[e] < st.shape[1 + e] - 3 for e in range(3)):
                assert not np.isfinite(got[(f,) + tuple(q)])


@pytest.mark.parametrize("n", [(4, 4, 4), (5, 7, 33), (32, 8, 8), (17, 15, 1 + 8)])
@pytest.mark.parametrize("r_excise", [0.3, 50.0])
def test_norms_at_block_edges(n, r_excise):
    """Blocks of 256 points with a ragged end, an excised set that is empty
    (r_excise past the grid) or not; the bar of the norms' parity tests."""
    from paper_1111_3344_gb300.bssn import Evolution
    c, st = _case(n, 11, r_excise=r_excise, punctures=[(1.0, 0.02, -0.01, 0.03)])
    evo = Evolution(T.gpu_params(c))
    evo.set_punctures(c["punctures"])
    evo.set_state(st)
    want = O.constraints(T.oracle_cfg(c), st)[0]
    assert np.allclose(evo.constraints(), want, rtol=1e-12, atol=0)
    st[7, 4, 5, 4] = np.nan  # a NaN shows in the sums and the maxima of both sets that hold it
    evo.set_state(st)
    got = evo.constraints()
    assert np.isnan(got[:8]).any() and (r_excise > 10 or np.isnan(got[8:]).any())
    evo.close()


@pytest.mark.parametrize("n", [(8, 4, 4), (9, 5, 5), (7, 4, 8), (16, 8, 4), (72, 20, 36),
                               (74, 21, 36), (64, 32, 60), (57, 58, 59)])
@pytest.mark.parametrize("conformal", ["W", "phi"])
def test_tile_form_equals_the_point_form(n, conformal):
    """The stage in tiles (csrc/k_stage_fx.cu; whole tiles, one point past them,
    one point short; with groups of threads up to 456 tiles, (72, 20, 36) being
    405 and (74, 21, 36) 540, without from there) against the oracle and against one point at a time, which
    a register that no tensor load can describe (8-byte aligned) takes: also
    with a field of zeros, fields that hold one tiny and one subnormal value
    (those tiles by the float64 sums), a shift of zero, and not a number in the padding of the rows.  Bars as above; the two forms differ
    by the roundings of both, twice the bar."""
    import torch
    from paper_1111_3344_gb300.bssn import Evolution
    c, st = _case(n, 23, conformal=conformal)
    if conformal == "phi":
        st[0] = -0.5 * np.log(st[0])
    st[21:24] = 0.0
    st[22, 4, 5, 4], st[23, 4, 5, 4] = 1e-290, 5e-324
    st[18:21, -6:] = 0.0
    evo = Evolution(T.gpu_params(c))
    reg = evo.numpy_to_register(st)
    reg.view(24, st.shape[1], st.shape[2], -1)[..., st.shape[3]:] = float("nan")  # the padding of a row may hold anything
    got = evo.register_to_numpy(evo.rhs(reg))
    odd = torch.empty(reg.numel() + 1, dtype=reg.dtype, device=reg.device)[1:].view(reg.shape)
    assert odd.data_ptr() % 16 == 8
    odd.copy_(reg)
    point = evo.register_to_numpy(evo.rhs(odd))
    evo.close()
    want, mag = O.rhs_mag(T.oracle_cfg(c), st)
    assert T.rounding_aware_errors(got, want, mag).max() <= 1.0
    assert T.rounding_aware_errors(point, want, mag).max() <= 1.0
    assert T.rounding_aware_errors(got, point, mag).max() <= 2.0


@pytest.mark.parametrize("n", [(16, 12, 8), (64, 40, 33)])
@pytest.mark.parametrize("precision", ["fp64", "ff"])
def test_captured_calls_equal_direct_ones(n, precision):
    """Steps and the right-hand side of a caller's register recorded into a graph
    (ordinary launches, the tensor map made during the capture) give the bits
    of the direct calls, whose launches overlap on the smaller grid; so does
    the context's own stream being the default one."""
    import torch
    from paper_1111_3344_gb300 import bssn as B
    c, st = _case(n, 29, precision=precision)
    evo = B.Evolution(T.gpu_params(c), stream=torch.cuda.Stream())
    evo.set_state(st)
    evo.rk4_step(3)
    want = evo.get_state()[0]
    reg = evo.numpy_to_register(st)
    torch.cuda.synchronize()
    out = torch.zeros_like(reg)
    B.bssn_rhs(evo.ctx, reg.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    out2 = torch.zeros_like(reg)
    evo.set_state(st)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=evo.stream):
        B.bssn_rhs(evo.ctx, reg.data_ptr(), out2.data_ptr())
        B.bssn_rk4_step(evo.ctx, 3)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, out2)
    assert np.array_equal(evo.get_state()[0], want)
    del graph
    evo.close()


@pytest.mark.parametrize("n", [(40, 40, 40), (33, 50, 61), (48, 45, 47), (24, 24, 24)])
@pytest.mark.parametrize("boundary", ["sommerfeld", "periodic"])
def test_mixed_tile_widths_give_the_same_bits(n, boundary):
    """The eleven-field mixed stage on 16-wide tiles (the first three grids, whole
    and partial ones) and 32-wide ones against the fused kernel: the same
    per-point operations, so the same bits (csrc/k_stage_tma.cu)."""
    from paper_1111_3344_gb300 import bssn as B
    c, st = _case(n, 31, precision="mixed", w_fp64_threshold=0.9)
    c["boundary"] = boundary
    names = [B.bssn_tile_name(q) for q in range(B.bssn_tile_count())]
    out = []
    for tile in ("tma11_32x8x1/1", "32x8x1/1"):
        evo = B.Evolution(T.gpu_params(c))
        B.bssn_set_tile(evo.ctx, names.index(tile))
        evo.set_state(st)
        evo.rk4_step(2)
        out.append(evo.get_state()[0])
        evo.close()
    assert np.isfinite(out[0]).all() and np.array_equal(out[0], out[1])
