"""The work a user has this framework do, as cases that can be timed and
compared: RK4 steps of single evolutions in each precision, one right-hand
side of a caller's state, batches of binaries, and the monitors of an output
step.  Sizes are those of the repository's own workloads (24^3 gauge wave,
128^3 and 256^3 puncture, binaries on 48^3 .. 128^3) and of its ragged tests.

States are Brill-Lindquist punctures (or a gauge wave) plus smooth seeded
low-mode perturbations of all 24 fields, so that every term of the equations
is non-zero, as it is a few steps into an evolution.

exact() restates the scheme in plain float64 torch: 4th-order stencils,
lopsided advection, Kreiss-Oliger dissipation, the Sommerfeld layers, classical
RK4, constraint norms, ADM integrals and Psi4.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1111_3344_gb300 import bssn as B

NF, GH = 24, 3
CHI, GT, TRK, AT, GAM, ALP, BETA, BB = 0, 1, 7, 8, 14, 17, 18, 21
SYM = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
PAIRS = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


# ------------------------------------------------------------------- cases
def _step(name, n, half, precision="fp64", boundary="sommerfeld", conformal="W", slicing="1+log", nsteps=1, q_R=0.0,
          data="bl", matter=False, what="step"):
    c = {"what": what, "nx": n[0], "ny": n[1], "nz": n[2], "half": half, "precision": precision,
         "boundary": boundary, "conformal": conformal, "slicing": slicing, "q_R": q_R, "nsteps": nsteps, "data": data,
         "matter": matter}
    return dict(c, name=name) if name else c


def _batch(name, precision, sizes, nsteps):
    c = {"what": "batch", "precision": precision, "sizes": ",".join(str(s) for s in sizes), "nsteps": nsteps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest evolution in use: the periodic gauge wave of the
        # convergence test, where launches and one block's latency count
        _step("wave24_fp64", (24, 24, 24), 0.5, boundary="periodic", data="wave"),
        # the headline: one step of the 128^3 puncture in float64
        _step("puncture128_fp64", (128, 128, 128), 8.0),
        # a production grid that fits no tile: odd sizes, the phi variant,
        # harmonic slicing, shift damping that falls off with radius
        _step("ragged_phi_fp64", (75, 53, 61), 6.0, conformal="phi", slicing="harmonic", q_R=3.0),
        # a caller's own integrator: one float64 right-hand side of its state,
        # with a stress-energy tensor
        _step("rhs80_matter_fp64", (80, 80, 80), 6.0, matter=True, what="rhs"),
        # quick-look evolutions in mixed precision, small and headline size
        _step("puncture48_mixed", (48, 48, 48), 6.0, precision="mixed"),
        _step("puncture128_mixed", (128, 128, 128), 8.0, precision="mixed"),
        # the largest single evolution of the precision study
        _step("puncture256_mixed", (256, 256, 256), 8.0, precision="mixed"),
        # double-word precision: the headline grid, and one that fits no tile
        _step("puncture128_ff", (128, 128, 128), 8.0, precision="ff"),
        _step("ragged_ff", (66, 57, 50), 6.0, precision="ff"),
        # several binaries advanced together and read back, as the batched
        # study and the server do
        _batch("batch_fp64", "fp64", (48, 64, 48, 96), 20),
        _batch("batch_mixed", "mixed", (48, 64, 48, 96, 64, 48), 100),
        # an output step: constraint norms, ADM integrals and Psi4
        _step("monitors128", (128, 128, 128), 8.0, what="monitors"),
    ]


def draw(rng):
    what = rng.choice(["step"] * 6 + ["rhs", "rhs", "batch", "monitors"])
    precision = rng.choice(["fp64", "fp64", "mixed", "ff"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if what == "batch":
        sizes = [rng.choice([32, 37, 48, 56, 64, 96]) for _ in range(rng.randint(2, 5))]
        points = sum(s ** 3 for s in sizes)
        rate = {"fp64": 70e6, "mixed": 450e6, "ff": 90e6}[precision]
        return _batch(None, precision, sizes, max(1, min(100, int(0.3 * rate / points))))
    n = [size(16, 160) for _ in range(3)]
    if rng.random() < 0.4:  # whole tiles
        n = [max(32, 32 * round(n[0] / 32)), max(8, 8 * round(n[1] / 8)), n[2]]
    boundary = rng.choice(["sommerfeld", "sommerfeld", "periodic"]) if what == "step" else "sommerfeld"
    return _step(None, n, rng.choice([4.0, 6.0, 8.0]), precision="fp64" if what != "step" else precision,
                 boundary=boundary, conformal=rng.choice(["W", "W", "phi"]),
                 slicing=rng.choice(["1+log", "1+log", "harmonic"]), nsteps=rng.choice([1, 1, 2]) if what == "step" else 1,
                 q_R=rng.choice([0.0, 3.0]), data="wave" if boundary == "periodic" else "bl",
                 matter=what == "rhs" and rng.random() < 0.5, what=what)


# ------------------------------------------------------------------ inputs
def _grid(case):
    """n, xmin, h of a single evolution: cubic cells, the longest axis on [-half, half]."""
    n = (case["nx"], case["ny"], case["nz"])
    h = 2.0 * case["half"] / max(n)
    # a cell corner at the origin, so that no point coincides with a puncture
    return n, tuple(-(m // 2) * h for m in n), h


def _coords(n, xmin, h):
    x = [xmin[d] + (torch.arange(n[d] + 2 * GH, dtype=torch.float64, device="cuda") - GH + 0.5) * h for d in range(3)]
    return x[0][None, None, :], x[1][None, :, None], x[2][:, None, None]


def _smooth(rng, X, Y, Z, size, periodic, amp):
    """A few seeded plane waves; periodic ones are whole waves along every axis."""
    f = torch.zeros(torch.broadcast_shapes(X.shape, Y.shape, Z.shape), dtype=torch.float64, device="cuda")
    for _ in range(3):
        k = rng.randint(-2, 3, size=3) if periodic else rng.uniform(-2.0, 2.0, size=3)
        ph, a = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(-1.0, 1.0)
        k = [2.0 * math.pi * k[d] / size[d] for d in range(3)]
        f += (a * amp / 3.0) * torch.sin(k[0] * X + k[1] * Y + k[2] * Z + ph)
    return f


def _state(n, xmin, h, data, conformal, punctures, seed):
    """(24, Z, Y, X) float64 state on every stored point."""
    rng = np.random.RandomState(seed % (1 << 31))
    X, Y, Z = _coords(n, xmin, h)
    shape = torch.broadcast_shapes(X.shape, Y.shape, Z.shape)
    st = torch.zeros((NF,) + tuple(shape), dtype=torch.float64, device="cuda")
    st[[GT, GT + 3, GT + 5]] = 1.0
    periodic = data == "wave"
    if periodic:  # gauge wave ds^2 = H (-dt^2 + dx^2) + dy^2 + dz^2 at t = 0
        A, d = 0.01 * rng.uniform(0.5, 1.5), n[0] * h
        H = (1.0 - A * torch.sin(2.0 * math.pi * X / d)).expand(shape)
        cb = H ** (1.0 / 3.0)
        st[CHI] = 1.0 / torch.sqrt(cb)
        st[GT], st[GT + 3], st[GT + 5] = H / cb, 1.0 / cb, 1.0 / cb
        Kxx = (-math.pi * A / d) * torch.cos(2.0 * math.pi * X / d).expand(shape) / torch.sqrt(H)
        st[TRK] = Kxx / H
        st[AT] = (Kxx - H * st[TRK] / 3.0) / cb
        st[AT + 3] = st[AT + 5] = -st[TRK] / (3.0 * cb)
        dH = (-2.0 * math.pi * A / d) * torch.cos(2.0 * math.pi * X / d).expand(shape)
        st[GAM] = (2.0 / 3.0) * dH / H ** (5.0 / 3.0)
        st[ALP] = torch.sqrt(H)
    else:
        psi = torch.ones(shape, dtype=torch.float64, device="cuda")
        for m, x, y, z in punctures:
            psi += 0.5 * m / torch.sqrt((X - x) ** 2 + (Y - y) ** 2 + (Z - z) ** 2)
        st[CHI] = psi ** -2
        st[ALP] = psi ** -2
    size = [n[d] * h for d in range(3)]
    amp = 1e-3 if periodic else 0.01
    for f in range(NF):
        p = _smooth(rng, X, Y, Z, size, periodic, amp)
        st[f] = st[f] * (1.0 + p) if f in (CHI, ALP) else st[f] + p
    if conformal == "phi":
        st[CHI] = -0.5 * torch.log(st[CHI])
    return st


def _punctures(case, seed):
    if case["data"] == "wave":
        return []
    rng = np.random.RandomState(seed % (1 << 31) + 7)
    return [(float(rng.uniform(0.8, 1.2)), 0.0, 0.0, 0.0)]


def _tmunu(n, xmin, h, seed):
    rng = np.random.RandomState(seed % (1 << 31) + 13)
    X, Y, Z = _coords(n, xmin, h)
    size = [n[d] * h for d in range(3)]
    t = [0.01 * (1.0 + _smooth(rng, X, Y, Z, size, False, 0.5))]
    t += [_smooth(rng, X, Y, Z, size, False, 0.005) for _ in range(9)]
    return torch.stack(t)


def _params(case, n, xmin, h):
    return B.Params(n=n, xmin=xmin, h=h, boundary=case["boundary"], conformal=case["conformal"],
                    slicing=case["slicing"], eta=2.0, q_R=case["q_R"] or math.inf, ko_eps=0.1, dt=0.25 * h,
                    precision=case["precision"], r_excise=1.0)


def _members(case, seed):
    """Binaries of a batch: masses, separations and domains as the batched workload draws them."""
    rng = np.random.RandomState(seed % (1 << 31) + 29)
    out = []
    for n in (int(s) for s in case["sizes"].split(",")):
        m1, m2 = rng.uniform(0.3, 0.7, size=2)
        s = rng.uniform(2.0, 6.0)
        L = max(8.0, 2.0 * s) * (m1 + m2)
        h = 2.0 * L / n
        xs = [round(v / h + 0.5 * (n % 2)) * h - 0.5 * h * (n % 2) for v in (s * m2 / (m1 + m2), -s * m1 / (m1 + m2))]
        y = 0.5 * h * (n % 2)
        out.append(((n, n, n), (-L,) * 3, h, [(m1, xs[0], y, y), (m2, xs[1], y, y)]))
    return out


_BATCH = {"boundary": "sommerfeld", "conformal": "W", "slicing": "1+log", "q_R": 0.0}


def prepare(case, seed):
    if case["what"] == "batch":
        members, c = _members(case, seed), dict(case, **_BATCH)
        params = [_params(c, *m[:3]) for m in members]
        b = B.Batch(case["precision"], pool_bytes=sum(B.Batch.member_bytes(p) for p in params) + (32 << 20),
                    max_members=len(members))
        ids = [b.add(p) for p in params]
        for q, (m, p) in enumerate(zip(ids, members)):
            b.set_state(m, _state(*p[:3], "bl", "W", p[3], seed + q).cpu().numpy())
        return {"batch": b, "ids": ids, "nsteps": case["nsteps"]}
    n, xmin, h = _grid(case)
    punct = _punctures(case, seed)
    evo = B.Evolution(_params(case, n, xmin, h))
    evo.set_initial_data("flat")
    evo.set_punctures(punct)
    evo.state_view()[..., : n[0] + 2 * GH] = _state(n, xmin, h, case["data"], case["conformal"], punct, seed)
    if case["matter"]:
        evo.set_matter(_tmunu(n, xmin, h, seed).cpu().numpy())
    s = {"evo": evo, "what": case["what"], "nsteps": case["nsteps"], "sx": n[0] + 2 * GH}
    if case["what"] == "monitors":
        s["psi4"] = evo.psi4()
    return s


def run(state):
    if "batch" in state:
        b = state["batch"]
        b.step(state["nsteps"])
        return [b.get_state(m)[0] for m in state["ids"]]
    evo = state["evo"]
    if state["what"] == "step":
        evo.rk4_step(state["nsteps"])
        return evo.state_view()[..., : state["sx"]]
    lay = evo.layout
    if state["what"] == "rhs":
        reg = evo.rhs()
        return reg.view(NF, lay["stored"][2], lay["stored"][1], lay["pitch"])[..., : state["sx"]]
    psi = evo.psi4(state["psi4"])
    return {"norms": evo.constraints(), "integrals": evo.adm_integrals()[0],
            "psi4": psi.view(2, lay["stored"][2], lay["stored"][1], lay["pitch"])[..., : state["sx"]]}


# -------------------------------------------------------------------- work
# Operations of one right-hand side at a point in the arrangement that the
# float64 kernels need least for (first and second differences, advection and
# dissipation of 24 fields, Christoffel symbols, Ricci tensor, the equations).
RHS_FLOPS = 3266.0
# ADM fields, curvature and constraints; R and the ADM integrands; Psi4
MONITOR_FLOPS = 1500.0 + 1300.0 + 2100.0


def work(case):
    if case["what"] == "batch":
        points = sum(int(s) ** 3 for s in case["sizes"].split(","))
        stored = sum((int(s) + 2 * GH) ** 3 for s in case["sizes"].split(","))
        per = {"fp64": 8.0, "mixed": 4.0, "ff": 8.0}[case["precision"]]
        # each step reads the state and writes the new one; the states come back to the host
        return {"bytes": case["nsteps"] * 2.0 * NF * per * stored + 8.0 * NF * stored,
                "flops": 4.0 * RHS_FLOPS * points * case["nsteps"]}
    n = (case["nx"], case["ny"], case["nz"])
    points = float(n[0]) * n[1] * n[2]
    stored = float(n[0] + 2 * GH) * (n[1] + 2 * GH) * (n[2] + 2 * GH)
    if case["what"] == "monitors":
        return {"bytes": 8.0 * (3 * NF * stored + 2 * points), "flops": MONITOR_FLOPS * points}
    if case["what"] == "rhs":
        return {"bytes": 8.0 * stored * (2 * NF + (10 if case["matter"] else 0)), "flops": RHS_FLOPS * points}
    # one step: y_n read and written once, as float64
    return {"bytes": case["nsteps"] * 2.0 * NF * 8.0 * stored, "flops": case["nsteps"] * 4.0 * RHS_FLOPS * points}


# ------------------------------------------------------------------- exact
class _Stencils:
    """Differences of a stored field at the interior points, spacing h."""

    def __init__(self, n, h):
        self.n, self.h = n, h

    def at(self, f, dx=0, dy=0, dz=0):
        n = self.n
        return f[..., GH + dz: GH + dz + n[2], GH + dy: GH + dy + n[1], GH + dx: GH + dx + n[0]]

    def shift(self, f, d, m, e=0, q=0):
        o = [0, 0, 0]
        o[d] += m
        o[e] += q
        return self.at(f, *o)

    def d1(self, f, d):
        s = self.shift
        return ((s(f, d, -2) - s(f, d, 2)) + 8.0 * (s(f, d, 1) - s(f, d, -1))) / (12.0 * self.h)

    def d2(self, f, a, b):
        s = self.shift
        if a == b:
            return (16.0 * (s(f, a, 1) + s(f, a, -1)) - (s(f, a, 2) + s(f, a, -2)) - 30.0 * s(f, a, 0)) / (12.0 * self.h ** 2)

        def line(m):
            return 8.0 * (s(f, a, m, b, 1) - s(f, a, m, b, -1)) - (s(f, a, m, b, 2) - s(f, a, m, b, -2))

        return (8.0 * (line(1) - line(-1)) - (line(2) - line(-2))) / (144.0 * self.h ** 2)

    def up(self, f, d, beta):
        s = self.shift
        p = -3.0 * s(f, d, -1) - 10.0 * s(f, d, 0) + 18.0 * s(f, d, 1) - 6.0 * s(f, d, 2) + s(f, d, 3)
        m = -3.0 * s(f, d, 1) - 10.0 * s(f, d, 0) + 18.0 * s(f, d, -1) - 6.0 * s(f, d, -2) + s(f, d, -3)
        return torch.where(beta >= 0.0, p, -m) / (12.0 * self.h)

    def ko(self, f, d):
        s = self.shift
        return (s(f, d, 3) + s(f, d, -3)) - 6.0 * (s(f, d, 2) + s(f, d, -2)) + 15.0 * (s(f, d, 1) + s(f, d, -1)) - 20.0 * s(f, d, 0)


def _mat(v):
    return [[v[SYM[a][b]] for b in range(3)] for a in range(3)]


def _inverse(g):
    c = [g[1][1] * g[2][2] - g[1][2] * g[1][2], g[0][2] * g[1][2] - g[0][1] * g[2][2], g[0][1] * g[1][2] - g[0][2] * g[1][1]]
    det = g[0][0] * c[0] + g[0][1] * c[1] + g[0][2] * c[2]
    u = [c[0], c[1], c[2], g[0][0] * g[2][2] - g[0][2] ** 2, g[0][1] * g[0][2] - g[0][0] * g[1][2], g[0][0] * g[1][1] - g[0][1] ** 2]
    return _mat([v / det for v in u]), det


def _christoffel(dg, gu):
    G1 = [_mat([0.5 * (dg[a][SYM[k][b]] + dg[b][SYM[k][a]] - dg[k][SYM[a][b]]) for a, b in PAIRS]) for k in range(3)]
    G2 = [_mat([sum(gu[k][l] * G1[l][a][b] for l in range(3)) for a, b in PAIRS]) for k in range(3)]
    return G1, G2


def _conformal_ricci(g, gu, dg, ddg, dG, G1, G2):
    """Rt_ij (pairs) with the evolved Gt in gt_k(i d_j) Gt^k only; dgu[k] = d_l gt^{lk}."""
    dgu = [-sum(gu[l][a] * gu[k][b] * dg[l][SYM[a][b]] for l in range(3) for a in range(3) for b in range(3)) for k in range(3)]
    R = []
    for a, b in PAIRS:
        s = sum(-0.5 * gu[k][l] * ddg[SYM[k][l]][SYM[a][b]] for k in range(3) for l in range(3))
        s = s + sum(0.5 * (g[k][a] * dG[b][k] + g[k][b] * dG[a][k]) for k in range(3))
        s = s - sum(0.5 * (G1[a][b][k] + G1[b][a][k]) * dgu[k] for k in range(3))
        for l in range(3):
            for m in range(3):
                s = s + gu[l][m] * sum(G2[k][l][a] * G1[b][k][m] + G2[k][l][b] * G1[a][k][m] + G2[k][a][m] * G1[k][l][b]
                                       for k in range(3))
        R.append(s)
    return R, dgu


def _matter(S, T, alp, beta):
    t = [S.at(T[q]) for q in range(10)]
    Sij = _mat(t[4:])
    E = t[0] - 2.0 * sum(beta[a] * t[1 + a] for a in range(3)) + sum(beta[a] * beta[b] * Sij[a][b] for a in range(3) for b in range(3))
    Si = [-(t[1 + a] - sum(beta[b] * Sij[b][a] for b in range(3))) / alp for a in range(3)]
    return E / alp ** 2, Si, Sij


def _interior_rhs(st, n, xmin, h, use_w, slicing, q_R, T):
    S = _Stencils(n, h)
    v = [S.at(st[f]) for f in range(NF)]
    chi, trK, alp, beta, Bv = v[CHI], v[TRK], v[ALP], v[BETA:BETA + 3], v[BB:BB + 3]
    g, A = _mat(v[GT:GT + 6]), _mat(v[AT:AT + 6])
    gu, _ = _inverse(g)
    dg = [[S.d1(st[GT + m], d) for m in range(6)] for d in range(3)]
    ddg = [[S.d2(st[GT + m], a, b) for m in range(6)] for a, b in PAIRS]
    dG = [[S.d1(st[GAM + a], d) for a in range(3)] for d in range(3)]
    G1, G2 = _christoffel(dg, gu)
    Rt, dgu = _conformal_ricci(g, gu, dg, ddg, dG, G1, G2)
    del ddg, G1
    db = [[S.d1(st[BETA + a], d) for a in range(3)] for d in range(3)]
    dchi, dalp, dK = ([S.d1(st[f], d) for d in range(3)] for f in (CHI, ALP, TRK))
    ddchi, ddalp = ([S.d2(st[f], a, b) for a, b in PAIRS] for f in (CHI, ALP))
    if use_w:
        Wd = chi.clamp_min(1e-10)
        em4 = chi * chi
        dphi = [-d / (2.0 * Wd) for d in dchi]
        ddphi = [-ddchi[q] / (2.0 * Wd) + dchi[a] * dchi[b] / (2.0 * Wd * Wd) for q, (a, b) in enumerate(PAIRS)]
    else:
        em4, dphi, ddphi = torch.exp(-4.0 * chi), dchi, ddchi
    DDphi = [ddphi[q] - sum(G2[k][a][b] * dphi[k] for k in range(3)) for q, (a, b) in enumerate(PAIRS)]
    DDalp = [ddalp[q] - sum(G2[k][a][b] * dalp[k] for k in range(3)) for q, (a, b) in enumerate(PAIRS)]

    def contract(x):
        return sum(gu[a][b] * x[SYM[a][b]] for a in range(3) for b in range(3))

    lap_phi, lap_alp = contract(DDphi), contract(DDalp)
    grad2 = sum(gu[a][b] * dphi[a] * dphi[b] for a in range(3) for b in range(3))
    cross = sum(gu[a][b] * dphi[a] * dalp[b] for a in range(3) for b in range(3))
    Xf = []
    for q, (a, b) in enumerate(PAIRS):
        rphi = -2.0 * DDphi[q] - 2.0 * g[a][b] * lap_phi + 4.0 * dphi[a] * dphi[b] - 4.0 * g[a][b] * grad2
        Xf.append(alp * (Rt[q] + rphi) - DDalp[q] + 2.0 * (dphi[a] * dalp[b] + dphi[b] * dalp[a]))
    trX = contract(Xf)
    Aud = [[sum(gu[a][l] * A[l][b] for l in range(3)) for b in range(3)] for a in range(3)]
    Auu = [[sum(Aud[a][l] * gu[l][b] for l in range(3)) for b in range(3)] for a in range(3)]
    AA = sum(Auu[a][b] * A[a][b] for a in range(3) for b in range(3))
    divb = db[0][0] + db[1][1] + db[2][2]
    r = [None] * NF
    r[CHI] = (chi / 3.0) * (alp * trK - divb) if use_w else (divb - alp * trK) / 6.0
    r[TRK] = -em4 * (lap_alp + 2.0 * cross) + alp * (AA + trK * trK / 3.0)
    if T is not None:
        E, Si, Sij = _matter(S, T, alp, beta)
        trs = sum(gu[a][b] * Sij[a][b] for a in range(3) for b in range(3))
        r[TRK] = r[TRK] + 4.0 * math.pi * alp * (E + em4 * trs)
    for q, (a, b) in enumerate(PAIRS):
        r[GT + q] = -2.0 * alp * A[a][b] + sum(g[k][a] * db[b][k] + g[k][b] * db[a][k] for k in range(3)) - (2.0 / 3.0) * g[a][b] * divb
        s = em4 * (Xf[q] - g[a][b] * trX / 3.0) + alp * trK * A[a][b] - (2.0 / 3.0) * A[a][b] * divb
        s = s - 2.0 * alp * sum(A[a][k] * Aud[k][b] for k in range(3)) + sum(A[k][a] * db[b][k] + A[k][b] * db[a][k] for k in range(3))
        if T is not None:
            s = s - 8.0 * math.pi * alp * em4 * (Sij[a][b] - g[a][b] * trs / 3.0)
        r[AT + q] = s
    ddb = [[S.d2(st[BETA + c], a, b) for c in range(3)] for a, b in PAIRS]
    x = [xmin[d] + (torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * h for d in range(3)]
    rr = torch.sqrt(x[0][None, None, :] ** 2 + x[1][None, :, None] ** 2 + x[2][:, None, None] ** 2)
    damp = 2.0 if not q_R else 2.0 * torch.where(rr <= q_R, torch.ones_like(rr), q_R / rr)
    for a in range(3):
        s = sum(gu[k][l] * ddb[SYM[k][l]][a] for k in range(3) for l in range(3))
        s = s + sum(gu[a][j] * ddb[SYM[j][k]][k] for j in range(3) for k in range(3)) / 3.0
        s = s + sum(dgu[j] * db[j][a] for j in range(3)) - (2.0 / 3.0) * dgu[a] * divb
        s = s - 2.0 * sum(Auu[a][j] * dalp[j] for j in range(3))
        br = sum(-(2.0 / 3.0) * gu[a][j] * dK[j] + 6.0 * Auu[a][j] * dphi[j] for j in range(3))
        br = br + sum(G2[a][k][l] * Auu[k][l] for k in range(3) for l in range(3))
        s = s + 2.0 * alp * br
        if T is not None:
            s = s - 16.0 * math.pi * alp * sum(gu[a][j] * Si[j] for j in range(3))
        r[GAM + a] = s
        r[BETA + a] = 0.75 * Bv[a]
        r[BB + a] = s - damp * Bv[a]
    r[ALP] = -2.0 * alp * trK if slicing == "1+log" else (-alp * alp * trK if slicing == "harmonic" else torch.zeros_like(alp))
    del ddb, ddalp, ddchi, DDphi, DDalp, Xf, Rt
    for f in range(NF):
        adv = sum(beta[d] * S.up(st[f], d, beta[d]) for d in range(3))
        r[f] = r[f] + adv + (0.1 / (64.0 * h)) * (S.ko(st[f], 0) + S.ko(st[f], 1) + S.ko(st[f], 2))
    return torch.stack(r)


def _radiative(f, X, Y, Z, r, h, x0, v0):
    def diff(dim):
        m = f.shape[dim]

        def at(a, b):
            return f.narrow(dim, a, b - a)

        d = torch.empty_like(f)
        d.narrow(dim, 1, m - 2).copy_((at(2, m) - at(0, m - 2)) / (2.0 * h))
        d.narrow(dim, 0, 1).copy_(-(3.0 * at(0, 1) - 4.0 * at(1, 2) + at(2, 3)) / (2.0 * h))
        d.narrow(dim, m - 1, 1).copy_((3.0 * at(m - 1, m) - 4.0 * at(m - 2, m - 1) + at(m - 3, m - 2)) / (2.0 * h))
        return d

    return -v0 * (X * diff(2) + Y * diff(1) + Z * diff(0)) / r - v0 * (f - x0) / r


def _rhs(st, n, xmin, h, use_w, slicing, q_R, periodic, T=None):
    """The right-hand side on every stored point (ghosts: 0 when periodic)."""
    k = _interior_rhs(st, n, xmin, h, use_w, slicing, q_R, T)
    inner = (slice(GH, GH + n[2]), slice(GH, GH + n[1]), slice(GH, GH + n[0]))
    out = torch.zeros_like(st)
    if not periodic:
        X, Y, Z = _coords(n, xmin, h)
        r = torch.sqrt(X * X + Y * Y + Z * Z)
        near = [torch.clamp(torch.arange(n[d] + 2 * GH, device="cuda"), GH, GH + n[d] - 1) for d in (2, 1, 0)]

        def anchored(a):  # each point's nearest interior point
            return a[near[0]][:, near[1]][:, :, near[2]]

        fac = (anchored(r) / r) ** 2
        for f in range(NF):
            one = f in (ALP, GT, GT + 3, GT + 5) or (f == CHI and use_w)
            rad = _radiative(st[f], X, Y, Z, r, h, 1.0 if one else 0.0, math.sqrt(2.0) if f in (ALP, TRK) else 1.0)
            e = torch.zeros_like(rad)
            e[inner] = k[f] - rad[inner]
            out[f] = rad + fac * anchored(e)
    out[(slice(None),) + inner] = k
    return out


def _fill_periodic(st, n):
    for dim, m in ((3, n[0]), (2, n[1]), (1, n[2])):
        st.narrow(dim, 0, GH).copy_(st.narrow(dim, m, GH).clone())
        st.narrow(dim, GH + m, GH).copy_(st.narrow(dim, GH, GH).clone())


def _rk4(st, n, xmin, h, use_w, slicing, q_R, periodic, nsteps):
    dt = 0.25 * h
    for _ in range(nsteps):
        if periodic:
            _fill_periodic(st, n)
        y, acc = st, None
        for q, (a, w) in enumerate(((0.5, 1.0), (0.5, 2.0), (1.0, 2.0), (0.0, 1.0))):
            k = _rhs(y, n, xmin, h, use_w, slicing, q_R, periodic)
            acc = k.clone() if acc is None else acc.add_(k, alpha=w)
            if q < 3:
                y = st + (a * dt) * k
                if periodic:
                    _fill_periodic(y, n)
        st = st + (dt / 6.0) * acc
        if periodic:
            _fill_periodic(st, n)
    return st


def _outside(n, xmin, h, punctures):
    x = [xmin[d] + (torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * h for d in range(3)]
    keep = torch.ones((n[2], n[1], n[0]), dtype=torch.bool, device="cuda")
    for _, px, py, pz in punctures:
        keep &= torch.sqrt((x[0][None, None, :] - px) ** 2 + (x[1][None, :, None] - py) ** 2 + (x[2][:, None, None] - pz) ** 2) > 1.0
    return keep


def _monitors(st, n, xmin, h, use_w, punctures):
    S = _Stencils(n, h)
    x = [xmin[d] + (torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * h for d in range(3)]
    x = [x[0][None, None, :].expand(n[2], n[1], n[0]), x[1][None, :, None].expand(n[2], n[1], n[0]),
         x[2][:, None, None].expand(n[2], n[1], n[0])]
    # ADM fields, formed pointwise and then differenced
    e4 = 1.0 / st[CHI] ** 2 if use_w else torch.exp(4.0 * st[CHI])
    gam = [e4 * st[GT + m] for m in range(6)]
    Kf = [e4 * (st[AT + m] + st[GT + m] * st[TRK] / 3.0) for m in range(6)]
    g, K = _mat([S.at(f) for f in gam]), _mat([S.at(f) for f in Kf])
    gu, det = _inverse(g)
    dg = [[S.d1(gam[m], d) for m in range(6)] for d in range(3)]
    dKf = [[S.d1(Kf[m], d) for m in range(6)] for d in range(3)]
    ddg = [[S.d2(gam[m], a, b) for m in range(6)] for a, b in PAIRS]
    _, G = _christoffel(dg, gu)
    trK = sum(gu[a][b] * K[a][b] for a in range(3) for b in range(3))
    Kud = [[sum(gu[a][l] * K[l][b] for l in range(3)) for b in range(3)] for a in range(3)]

    def riemann(a, b, c, d):
        s = 0.5 * (ddg[SYM[b][c]][SYM[a][d]] + ddg[SYM[a][d]][SYM[b][c]] - ddg[SYM[a][c]][SYM[b][d]] - ddg[SYM[b][d]][SYM[a][c]])
        return s + sum(g[m][p] * (G[m][b][c] * G[p][a][d] - G[m][b][d] * G[p][a][c]) for m in range(3) for p in range(3))

    R4 = [[[[riemann(a, b, c, d) for d in range(3)] for c in range(3)] for b in range(3)] for a in range(3)]
    Ric = [[sum(gu[a][c] * R4[a][b][c][d] for a in range(3) for c in range(3)) for d in range(3)] for b in range(3)]
    DK = [[[dKf[m][SYM[a][b]] - sum(G[l][m][a] * K[l][b] + G[l][m][b] * K[a][l] for l in range(3)) for b in range(3)]
           for a in range(3)] for m in range(3)]
    # constraints and their norms
    H = sum(gu[a][b] * Ric[a][b] for a in range(3) for b in range(3))
    H = H - sum(Kud[a][b] * Kud[b][a] for a in range(3) for b in range(3)) + trK * trK
    C = [H] + [sum(gu[j][k] * (DK[k][a][j] - DK[a][j][k]) for j in range(3) for k in range(3)) for a in range(3)]
    keep = _outside(n, xmin, h, punctures)
    norms = []
    for mask in (torch.ones_like(keep), keep):
        c = [v[mask] for v in C]
        norms += [float(torch.sqrt((v * v).mean())) for v in c] + [float(v.abs().max()) for v in c]
    # Psi4: triad by Gram-Schmidt in the order phi, r, theta
    rv, pv = list(x), [-x[1], x[0], torch.zeros_like(x[0])]
    eps = [(k, l, m, (k - l) * (l - m) * (m - k) / 2.0) for k in range(3) for l in range(3) for m in range(3) if len({k, l, m}) == 3]
    sdet = torch.sqrt(det)
    tv = [sdet * sum(e * gu[a][k] * pv[l] * rv[m] for k, l, m, e in eps) for a in range(3)]

    def dot(u, w):
        return sum(g[a][b] * u[a] * w[b] for a in range(3) for b in range(3))

    pp = dot(pv, pv)
    axis = ~(pp > 0.0)
    pv = [p / torch.sqrt(pp) for p in pv]
    rp = dot(rv, pv)
    rv = [rv[a] - rp * pv[a] for a in range(3)]
    rn = torch.sqrt(dot(rv, rv))
    rv = [v / rn for v in rv]
    tp, tr = dot(tv, pv), dot(tv, rv)
    tv = [tv[a] - tp * pv[a] - tr * rv[a] for a in range(3)]
    tn = torch.sqrt(dot(tv, tv))
    tv = [v / tn for v in tv]
    s2 = 1.0 / math.sqrt(2.0)
    nv = [-s2 * v for v in rv]
    # Q_bd of the curvature, contracted with mbar mbar = (theta - i phi)(theta - i phi)/2
    re, im = torch.zeros_like(pp), torch.zeros_like(pp)
    for b in range(3):
        for d in range(3):
            q = 0.5 * (Ric[b][d] + trK * K[b][d] - sum(K[b][m] * Kud[m][d] for m in range(3)))
            for a in range(3):
                q = q + 2.0 * s2 * (DK[a][b][d] - DK[d][b][a]) * nv[a]
                for c in range(3):
                    q = q + (R4[a][b][c][d] + K[a][c] * K[b][d] - K[a][d] * K[b][c]) * nv[a] * nv[c]
            re += 0.5 * q * (tv[b] * tv[d] - pv[b] * pv[d])
            im -= 0.5 * q * (tv[b] * pv[d] + pv[b] * tv[d])
    psi4 = torch.zeros((2,) + tuple(st.shape[1:]), dtype=torch.float64, device="cuda")
    for q, v in enumerate((re, im)):
        S.at(psi4[q]).copy_(torch.where(axis, torch.zeros_like(v), v))
    # ADM mass and angular momentum, from the conformal variables
    v = [S.at(st[f]) for f in range(NF)]
    ct, A = _mat(v[GT:GT + 6]), _mat(v[AT:AT + 6])
    cu, _ = _inverse(ct)
    dc = [[S.d1(st[GT + m], d) for m in range(6)] for d in range(3)]
    ddc = [[S.d2(st[GT + m], a, b) for m in range(6)] for a, b in PAIRS]
    dG = [[S.d1(st[GAM + a], d) for a in range(3)] for d in range(3)]
    dK = [S.d1(st[TRK], d) for d in range(3)]
    G1, G2 = _christoffel(dc, cu)
    Rt, _ = _conformal_ricci(ct, cu, dc, ddc, dG, G1, G2)
    ephi = 1.0 / torch.sqrt(v[CHI].clamp_min(1e-10)) if use_w else torch.exp(v[CHI])
    Aud = [[sum(cu[a][l] * A[l][b] for l in range(3)) for b in range(3)] for a in range(3)]
    Auu = [[sum(Aud[a][l] * cu[l][b] for l in range(3)) for b in range(3)] for a in range(3)]
    AA = sum(Auu[a][b] * A[a][b] for a in range(3) for b in range(3))
    trR = sum(cu[a][b] * Rt[SYM[a][b]] for a in range(3) for b in range(3))
    dens = [(ephi ** 5 * (AA - (2.0 / 3.0) * v[TRK] ** 2) - ephi * trR) / (16.0 * math.pi)]
    AdG = [-sum(Auu[a][b] * dc[k][SYM[a][b]] for a in range(3) for b in range(3)) for k in range(3)]
    for i in range(3):
        s = sum(e * (Aud[j][k] + (2.0 / 3.0) * x[j] * dK[k] - 0.5 * x[j] * AdG[k]) for q, j, k, e in eps if q == i)
        dens.append(ephi ** 6 * s / (8.0 * math.pi))
    integrals = [float(v.sum()) * h ** 3 for v in dens] + [float(v[keep].sum()) * h ** 3 for v in dens]
    return {"norms": np.array(norms), "integrals": np.array(integrals), "psi4": psi4}


def exact(case, seed):
    if case["what"] == "batch":
        if case["nsteps"] * len(case["sizes"].split(",")) > 80:  # too long for plain torch
            return None
        return [_rk4(_state(*m[:3], "bl", "W", m[3], seed + q), *m[:3], True, "1+log", 0.0, False, case["nsteps"])
                for q, m in enumerate(_members(case, seed))]
    n, xmin, h = _grid(case)
    punct, use_w = _punctures(case, seed), case["conformal"] == "W"
    st = _state(n, xmin, h, case["data"], case["conformal"], punct, seed)
    periodic = case["boundary"] == "periodic"
    if case["what"] == "step":
        return _rk4(st, n, xmin, h, use_w, case["slicing"], case["q_R"], periodic, case["nsteps"])
    if case["what"] == "rhs":
        return _rhs(st, n, xmin, h, use_w, case["slicing"], case["q_R"], periodic,
                    _tmunu(n, xmin, h, seed) if case["matter"] else None)
    return _monitors(st, n, xmin, h, use_w, punct)
