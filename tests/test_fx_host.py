"""The integer stencil arithmetic of csrc/fx.cuh and csrc/rhs_fx_tile.cuh compiled
for the host (the intrinsics they use restated below) and compared with exact
rational arithmetic: conversions, the weighted sum of stencil results over the
whole range of its weights, and a field's stencils in a tile's box, also at the
largest values that its sums may take.  Signed overflow aborts (-ftrapv).

Bars, from the bounds that the headers state: a conversion rounds to half a unit
or truncates to one; the weighted sum is off by 2^-56 of its largest product
and 2^-53 of itself; a derivative by half a unit a tap times the taps'
coefficients, the units its halvings drop, and 2^-53 of itself."""
import ctypes
import os
import random
import shutil
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1111_3344_gb300", "csrc")

SRC = r"""
#include <cuda_runtime.h>
#include <cstring>
#include <cmath>
using std::max;
using std::min;
static inline long long bits(double v) { long long b; memcpy(&b, &v, 8); return b; }
static inline int __double2hiint(double v) { return (int)(bits(v) >> 32); }
static inline int __double2loint(double v) { return (int)bits(v); }
static inline double __longlong_as_double(long long b) { double v; memcpy(&v, &b, 8); return v; }
static inline long long __double_as_longlong(double v) { return bits(v); }
static inline double __hiloint2double(int h, int l) { return __longlong_as_double((long long)(((unsigned long long)(unsigned)h << 32) | (unsigned)l)); }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline long long __mul64hi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
template <typename T> static inline T __ldg(const T* p) { return *p; }
using std::isinf;
#ifndef __noinline__
#define __noinline__
#endif
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
size_t __cvta_generic_to_shared(const void*);
int __syncthreads_and(int);
int __syncthreads_or(int);
void __syncthreads();
unsigned __reduce_max_sync(unsigned, unsigned);
#include "rhs_fx_tile.cuh"
using namespace bssn;
using Sh = FxTile<8, 4, 4>;
extern "C" {
long long h_from(double v, int E) { return fx_from(v, E); }
long long h_near(double v, int E) { return fx_near<FX_TILE_BITS>(v, E); }
double h_to(long long s, int E) { return fx_to(s, E); }
int h_weight(double v, long long* w) { return fx_weight(v, *w); }
double h_dot(const long long* a, int E, const long long* w) {
  const long long x[4] = {a[0], a[1], a[2], a[3]}, y[4] = {w[0], w[1], w[2], w[3]};
  return fx_dot(x, E, y);
}
int h_tile_bits() { return FX_TILE_BITS; }
// a box of values (BOX doubles) and 10 weights; out: r, 14 slots; the point at (i, j, k) of the tile
int h_stencils(const double* box, int q, const double* w4, const double* g6, const int* neg, int i, int j, int k,
               double* out) {
  static long long ib[Sh::BOX];
  static double wt[10 * Sh::THREADS];
  unsigned top = 0;
  for (int n = 0; n < Sh::BOX; n++) top = max(top, (unsigned)__double2hiint(box[n]) & 0x7fffffffu);
  const int E = max((int)(top >> 20), 256) + FX_BITS - FX_TILE_BITS;
  for (int n = 0; n < Sh::BOX; n++) ib[n] = fx_near<FX_TILE_BITS>(box[n], E + FX_TILE_BITS - FX_BITS);
  for (int d = 0; d < 4; d++) {
    long long x;
    if (!fx_weight(w4[d], x)) return -1;
    wt[(d < 3 ? d : 9) * Sh::THREADS] = __longlong_as_double(x);
  }
  for (int m = 0; m < 6; m++) wt[(3 + m) * Sh::THREADS] = g6[m];
  const long long* c = ib + ((k + GH) * Sh::BY + j + GH) * Sh::BX + i + GH;
  bool near = false;
  auto S = [&](int n) -> double& { return out[1 + n]; };
  out[0] = fx_stencils<Sh>(c, q, fx_order(q), fx_up(q), E, wt, neg, S, 0, near);
  return near;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not (shutil.which("g++") and os.path.exists(os.path.join(inc, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ftrapv", "-ffp-contract=off", "-w", "-fPIC", "-shared", "-I", inc,
                    "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    D, I, L = ctypes.c_double, ctypes.c_int, ctypes.c_longlong
    P = ctypes.POINTER
    for name, res, args in (("h_from", L, [D, I]), ("h_near", L, [D, I]), ("h_to", D, [L, I]), ("h_weight", I, [D, P(L)]),
                            ("h_dot", D, [P(L), I, P(L)]), ("h_tile_bits", I, []),
                            ("h_stencils", I, [P(D), I, P(D), P(D), P(I), I, I, I, P(D)])):
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    return lib


def unit(e):
    return Fr(2) ** e


def test_conversions(lib):
    rng = random.Random(1)
    bits = lib.h_tile_bits()
    for _ in range(4000):
        e = rng.randint(300, 1800)
        v = rng.choice([-1, 1]) * (1 + rng.random()) * 2.0 ** (e - 1023)
        E = e + rng.choice([0, 0, 1, 2, 3, 5, 30, 52, 53, 56, 57, 63, 64, 70, 200])
        assert abs(lib.h_from(v, E) - Fr(v) / unit(E - 1075 - 2)) < 1
        assert abs(lib.h_near(v, E) - Fr(v) / unit(E - 1075 - bits)) <= Fr(1, 2)
        assert abs(lib.h_near(v, E)) < 2 ** (53 + bits)
        s = rng.choice([-1, 1]) * rng.getrandbits(rng.randint(1, 63))
        got = Fr(lib.h_to(s, E))
        assert abs(got - s * unit(E - 1075 - 2)) <= abs(got) * unit(-53)
    assert lib.h_from(0.0, 900) == lib.h_near(-0.0, 900) == 0 and lib.h_to(0, 900) == 0.0


def test_weights_and_their_sum(lib):
    """Weights and stencil results of every size against one another, zeros among
    them, at both ends of the exponents that are taken."""
    rng = random.Random(2)
    L4 = ctypes.c_longlong * 4
    w1 = ctypes.c_longlong()
    for e, ok in ((894, 0), (895, 1), (1123, 1), (1124, 0), (0, 0), (2047, 0)):
        v = float(np.frombuffer(((e << 52) | 5).to_bytes(8, "little"), dtype=np.float64)[0])
        assert lib.h_weight(v, ctypes.byref(w1)) == ok
    assert lib.h_weight(0.0, ctypes.byref(w1)) == 1 and w1.value == 0
    for n in range(20000):
        E = rng.choice([254, 600, 1023, 1900])
        spread = rng.choice([3, 40, 228])
        lo = rng.randint(-128, 100 - spread)
        w = [0.0 if rng.random() < 0.15 else (1 + rng.random()) * 2.0 ** rng.randint(lo, lo + spread) for _ in range(4)]
        a = [0 if rng.random() < 0.15 else rng.choice([-1, 1]) * rng.getrandbits(rng.choice([1, 8, 40, 62, 63])) for _ in range(4)]
        if n % 7 == 0:
            a[rng.randrange(4)] = -1
        if n % 50 == 0:
            a = [-(2 ** 63) + 1 if x < 0 else 2 ** 63 - 1 for x in a]
        ws = L4()
        for q in range(4):
            assert lib.h_weight(w[q], ctypes.byref(w1)) == 1
            ws[q] = w1.value
        prod = [a[q] * Fr(w[q]) * unit(E - 1077) for q in range(4)]
        want, big = sum(prod), max(abs(p) for p in prod)
        got = Fr(lib.h_dot(L4(*a), E, ws))
        assert abs(got - want) <= big * unit(-56) + abs(want) * unit(-53) * Fr(3, 2), (a, w)


def _exact(box, q, c, bh, kap, neg):
    """(advection and dissipation, 12h d, 144 h^2 d d (xx xy xz yy yz zz)) of the box at c, exactly,
    and for each the sum of |coefficient|s of its taps."""
    def f(d):
        return Fr(float(box[tuple(c[n] + d[n] for n in range(3))]))

    def ax(a, m):
        d = [0, 0, 0]
        d[2 - a] = m
        return tuple(d)
    r = Fr(0)
    d1, dd = [], {}
    for a in range(3):
        v = {m: f(ax(a, m)) for m in range(-3, 4)}
        d1.append(8 * (v[1] - v[-1]) - (v[2] - v[-2]))
        dd[(a, a)] = 12 * (16 * (v[1] + v[-1]) - (v[2] + v[-2]) - 30 * v[0])
        K = 15 * (v[1] + v[-1]) - 6 * (v[2] + v[-2]) + (v[3] + v[-3]) - 20 * v[0]
        O = 21 * (v[1] - v[-1]) - 6 * (v[2] - v[-2]) + (v[3] - v[-3])
        r += Fr(bh[a]) * (K - O if neg[a] else K + O) + Fr(kap) * K
        for b in range(a + 1, 3):
            t = Fr(0)
            for m, cm in ((-2, 1), (-1, -8), (1, 8), (2, -1)):
                for n, cn in ((-2, 1), (-1, -8), (1, 8), (2, -1)):
                    t += cm * cn * f(tuple(x + y for x, y in zip(ax(a, m), ax(b, n))))
            dd[(a, b)] = t
    return r, d1, [dd[k] for k in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]


@pytest.mark.parametrize("kind", ["smooth", "wide", "largest", "small beside large"])
def test_stencils_in_a_box(lib, kind):
    rng = np.random.default_rng(5)
    bits = lib.h_tile_bits()
    for trial in range(12):
        box = rng.uniform(-1, 1, (10, 10, 14))
        if kind == "smooth":
            box = 1.0 + 1e-3 * box
        elif kind == "wide":
            box *= 10.0 ** rng.integers(-30, 1, box.shape)
        elif kind == "largest":  # every magnitude the largest of its exponent
            box = np.where(rng.random(box.shape) < 0.5, 1.0, -1.0) * np.nextafter(2.0, 0.0)
            if trial < 4:  # the signs that add up
                c = np.indices(box.shape).sum(0) % 2
                box = np.where(c == trial % 2, 1.0, -1.0) * np.nextafter(2.0, 0.0) * (1 if trial < 2 else -1)
        else:
            box *= 1e-6
            box[:, :, 11:] = 1.0
        i, j, k = int(rng.integers(0, 5)), int(rng.integers(0, 4)), int(rng.integers(0, 4))
        bh, kap = [float(x) for x in rng.uniform(0, 1, 3) * 10.0 ** rng.integers(-9, 2, 3)], 0.03
        neg = [int(x) for x in rng.integers(0, 2, 3) * -1]
        g6 = [float(x) for x in rng.uniform(0.5, 1.5, 6)]
        out = (ctypes.c_double * 16)()
        flat = np.ascontiguousarray(box)
        star = np.array([box[k + 3, j + 3, i + 3]] + [box[k + 3 + m * (a == 2), j + 3 + m * (a == 1), i + 3 + m * (a == 0)]
                                                      for a in range(3) for m in (-2, 2)])
        biggest = float(np.abs(box).max())
        u = unit(int(np.frexp(biggest)[1]) - 53 - bits)  # a unit of the box's integers
        for q in (0, 7, 9, 12, 14, 20):
            near = lib.h_stencils(flat.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), q, (ctypes.c_double * 4)(*bh, 2 * kap),
                                  (ctypes.c_double * 6)(*g6), (ctypes.c_int * 3)(*neg), i, j, k, out)
            # near: some star value of 2^52 units or more (a value one unit below may round up to it)
            assert near == (float(np.abs(star).max()) >= float(2 ** 52 * u)) or kind == "wide"
            r, d1, dd = _exact(box, q, (k + 3, j + 3, i + 3), bh, kap, neg)
            order, up = (2 if q < 6 or 8 < q < 14 else (1 if q < 15 else 0)), (Fr(1, 2) if q < 9 else 1)
            # r: 38 taps in half sums a weight and the quarters dropped, each half a unit
            rb = u * (sum(Fr(b) for b in bh) * 40 + Fr(kap) * (96 + 12))
            pmax = max([abs(Fr(b)) for b in bh] + [Fr(kap)]) * Fr(biggest) * 192
            assert abs(Fr(out[0]) - r) <= rb + pmax * unit(-56) + abs(r) * unit(-52)
            if order >= 1:
                for a in range(3):
                    assert abs(Fr(out[1 + a]) - up * d1[a]) <= up * (9 * u + abs(d1[a]) * unit(-53))
            if order == 2:
                e = [up * (Fr(12 * 32 + 16) if m in (0, 3, 5) else Fr(162 + 8)) * u + up * abs(dd[m]) * unit(-53) for m in range(6)]
                if q != 9:
                    lap = up * sum(Fr(g) * x for g, x in zip(g6, dd))
                    assert abs(Fr(out[4]) - lap) <= sum(Fr(g) * x for g, x in zip(g6, e)) + sum(
                        Fr(g) * up * abs(x) for g, x in zip(g6, dd)) * unit(-50)
                kept = {9: range(6), 12: (1, 3, 4)}.get(q, ())
                for n, m in enumerate(kept):
                    assert abs(Fr(out[5 + n]) - up * dd[m]) <= e[m]
