"""The float64 right-hand side is as exact beside large values as without them:
aligning a stencil's values to the largest among several (csrc/fx.cuh) or in a
tile's whole box (csrc/rhs_fx_tile.cuh) must not cost a derivative the bits by
which values that it does not use exceed its own.

Bars.  A stencil's values are held to 2^-53 of their largest or better and its sums
to a few 2^-53, so a point's right-hand side is off by some hundred times 2^-53 M,
M the oracle's magnitude of the same expression at the same point: 1e-12 M has
a factor of 30 to spare.  The grids run both forms of the stage in tiles (up to
456 tiles with groups of threads, from there without)."""
import numpy as np
import pytest

import cases as T
import oracle as O
from paper_1111_3344_gb300 import inputs

pytestmark = pytest.mark.gpu

GRIDS = [(24, 20, 16), (74, 21, 36), (64, 32, 32)]  # 60, 540 and 512 tiles


def _rhs(c, st, point_form=False):
    """One right-hand side; point_form: of a register that no tensor load can
    describe (8-byte aligned), which is taken one point at a time."""
    import torch
    from paper_1111_3344_gb300.bssn import Evolution
    evo = Evolution(T.gpu_params(c))
    reg = evo.numpy_to_register(st)
    if point_form:
        odd = torch.empty(reg.numel() + 1, dtype=reg.dtype, device=reg.device)[1:].view(reg.shape)
        odd.copy_(reg)
        reg = odd
    out = evo.register_to_numpy(evo.rhs(reg))
    evo.close()
    return out


def _interior(n):
    return np.array([(i, j, k) for k in range(3, 3 + n[2]) for j in range(3, 3 + n[1]) for i in range(3, 3 + n[0])],
                    dtype=np.int32)


@pytest.mark.parametrize("form", ["point", "tiles"])
@pytest.mark.parametrize("n", GRIDS[:2])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_large_values_three_points_away(n, axis, form):
    """A lapse that is 1e6 larger from some index of an axis on: three points
    before it only the advection and dissipation of the lapse itself read the
    large values; every other field's right-hand side does not."""
    c = dict(n=n, xmin=(-0.9, -1.1, -0.7), h=0.11, boundary="sommerfeld")
    st = inputs.random_state(43, n, c["xmin"], c["h"], amp=0.05)
    at = 3 + n[axis] // 2 + 1
    st[(17,) + tuple(slice(at, None) if 2 - d == axis else slice(None) for d in range(3))] += 1e6
    ijk = np.array([q for q in _interior(n) if q[axis] == at - 3], dtype=np.int32)
    cfg = T.oracle_cfg(c)
    want, mag = O.rhs_points_ext(cfg, st, ijk).T, O.rhs_points_mag(cfg, st, ijk)[1].T
    got = _rhs(c, st, form == "point")[:, ijk[:, 2], ijk[:, 1], ijk[:, 0]]
    assert (np.abs(got - want) <= 1e-12 * mag).all(), (np.abs(got - want) / mag).max(axis=1)


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("across,along,ko", [(0.3, 1e-9, 0.0), (0.3, 1e-30, 0.0), (0.0, 1e-20, 0.0), (0.3, 1e-42, 0.0),
                                              (1e-60, 1e-50, 0.0), (0.0, 1e-9, 0.2)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_small_shift_beside_a_large_one(n, across, along, ko, axis):
    """A lapse that varies along one axis, where the shift is much smaller than
    along the others, K = 0: d_0 alpha is the small shift's advection (and the
    dissipation), to a few roundings of its own products: eight of 2^-53 of
    |beta| / 24h times the upwind sum's 76 max|alpha|, and of eps / 64h times the
    dissipation's 64."""
    h = 0.11
    c = dict(n=n, xmin=(-0.9, -1.1, -0.7), h=h, boundary="sommerfeld", ko_eps=ko)
    cfg = T.oracle_cfg(c)
    st = O.initial_data(cfg, "flat", [])
    shape = [1, 1, 1]
    shape[2 - axis] = -1
    st[17] = (1.0 + 0.3 * np.sin(1.7 * cfg.coords(axis))).reshape(shape)
    for d in range(3):
        st[18 + d] = along if d == axis else across
    ijk = _interior(n)
    want = O.rhs_points_ext(cfg, st, ijk)[:, 17]
    got = _rhs(c, st)[17][ijk[:, 2], ijk[:, 1], ijk[:, 0]]
    bar = 8 * 2.0 ** -53 * 1.3 * (along * 76 / (24 * h) + ko * 3 * 64 / (64 * h))
    assert np.abs(got - want).max() <= bar and np.abs(want).max() > 1e3 * bar


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("conformal,precision", [("W", "fp64"), ("phi", "fp64"), ("W", "ff")])
def test_small_values_beside_large_ones(n, conformal, precision):
    """Fields of size 1e-9 with cubes of size 0.05 (three points) here and there:
    every point none of whose stencils reaches a cube, against the oracle in
    extended precision."""
    c = dict(n=n, xmin=(-0.9, -1.1, -0.7), h=0.11, boundary="sommerfeld", conformal=conformal, precision=precision)
    st = inputs.random_state(41, n, c["xmin"], c["h"], amp=0.05)
    if conformal == "phi":
        st[0] = -0.5 * np.log(st[0])
    big = np.zeros(st.shape[1:], dtype=bool)
    for k in range(7, n[2], 11):
        for j in range(5, n[1], 11):
            for i in range(6, n[0], 12):
                big[k:k + 3, j:j + 3, i:i + 3] = True
    for f in (2, 7, 8, 10, 13, 14, 16, 18, 19, 20, 22, 23):
        st[f] *= 2e-8
        st[f][big] += 0.05
    reach = np.zeros_like(big)
    offs = [(0, 0, m) for m in range(-3, 4)]
    offs = {tuple(np.roll(o, r)) for o in offs for r in range(3)}
    offs |= {tuple(np.roll((0, a, b), r)) for a in range(-2, 3) for b in range(-2, 3) for r in range(3)}
    for o in offs:
        reach |= np.roll(big, o, (0, 1, 2))
    ijk = np.array([q for q in _interior(n) if not reach[q[2], q[1], q[0]]], dtype=np.int32)
    assert 0.2 * np.prod(n) < len(ijk) < 0.95 * np.prod(n)
    cfg = T.oracle_cfg(c)
    want = O.rhs_points_ext(cfg, st, ijk).T
    mag = O.rhs_points_mag(cfg, st, ijk)[1].T
    got = _rhs(c, st)[:, ijk[:, 2], ijk[:, 1], ijk[:, 0]]
    assert (np.abs(got - want) <= 1e-12 * mag).all(), (np.abs(got - want) / mag).max(axis=1)
