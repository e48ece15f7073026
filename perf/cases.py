"""The framework's work as a user has it done: timed cases over the public entry points.

A pass of every case is a whole piece of a user's program through the C ABI
(``paper_1604_08159_gb300.binding``): the initial condition, some time steps
(or none: a snapshot of fields), and the read of the result into device
buffers.  Sizes follow the repository's workloads: finest lattices 128^2 to
4096^2, eps 1e-3 to 1e-4, Krylov dimensions to 31, FP64 and mixed precision,
DD orders 4, 6 and 8, both time schemes, the velocity-Exner form, the passive
scalar and batched ensembles of uneven members.

Results: an FP64 run returns its active lattice indices and values, in buffers
with room for every lattice point (zero beyond the active count); a mixed run, whose values are FP32, the reconstruction on its finest lattice as FP32
(the adaptive grid of a mixed run is not a whole-number result: a detail
within FP32 rounding of eps may fall either way).

``exact`` is the same method in plain torch FP64 over dense lattices.
"""

import math

import numpy as np
import torch

from paper_1604_08159_gb300 import binding as wrc
from paper_1604_08159_gb300.workloads import RunParams

SGS_OFF, SGS_DYNAMIC = 0, 2
ROSENBROCK, EXNER = 1, 1
CS = 0.17


def _case(name, kind, n0, J, eps, steps, **kw):
    c = {"kind": kind, "n0": n0, "J": J, "eps": eps, "steps": steps, "m": 30, "prec": "fp64", "order": 4,
         "sgs": True, "vortices": 2, "re": 5000.0, "scheme": "frozen", "members": 1, "jmin": J}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest run: an equal pair on 128^2 without subgrid model, as a parameter study
        # or a test suite starts by the hundred; launches and grid barriers are most of it
        _case("pair_128_fp64", "steps", 16, 3, 1e-3, 20, m=20, sgs=False),
        # a small mixed-precision request of three vortices, as the request server gets them
        _case("three_256_mixed", "steps", 32, 3, 1e-4, 16, prec="mixed", vortices=3, re=37440.0),
        # the ordinary run: the pair at 1024^2 with the dynamic subgrid model
        _case("pair_1024_fp64", "steps", 32, 5, 1e-4, 12),
        # the same lattice once the vortices have wound up: a field of many vortices, several
        # times the active points
        _case("field_1024_fp64", "steps", 32, 5, 1e-4, 8, vortices=24),
        # the paper's higher DD order (2p = 6) on the same run
        _case("pair_1024_dd6_fp64", "steps", 32, 5, 1e-4, 8, order=6),
        # the largest lattice, in the mixed mode it is meant for
        _case("three_4096_mixed", "steps", 32, 7, 1e-4, 12, prec="mixed", vortices=3, re=37440.0),
        # second order in time: the full Jacobian, a Poisson solve per Krylov vector
        _case("rosenbrock_512_fp64", "steps", 32, 4, 1e-4, 3, scheme="rosenbrock"),
        # omega and the water-vapour front carried together
        _case("vapour_1024_fp64", "scalar", 32, 5, 1e-4, 6),
        # the compressible velocity-Exner form of the pair
        _case("exner_1024_fp64", "exner", 32, 5, 1e-4, 6, sgs=False, scheme="rosenbrock"),
        # uneven ensembles advanced together: mixed (the ensemble's own precision) and FP64
        _case("ensemble_48_mixed", "ensemble", 32, 6, 1e-4, 10, prec="mixed", members=48, jmin=3),
        _case("ensemble_17_fp64", "ensemble", 32, 5, 1e-4, 6, members=17, jmin=3),
        # no step at all: a sampled field in, its transform, and the fields of a snapshot out
        _case("snapshot_2048_fp64", "snapshot", 32, 6, 1e-4, 0),
    ]


def draw(rng):
    kind = rng.choice(["fp64"] * 5 + ["mixed"] * 3 + ["rosenbrock", "scalar", "exner", "snapshot"] + ["ensemble"] * 3)
    eps = 10.0 ** rng.uniform(-4.0, -3.0)
    m = rng.randint(10, 31)
    order = rng.choice([4, 4, 4, 6, 8])
    re = 5000.0 * (37440.0 / 5000.0) ** rng.random()
    nv = rng.choice([2, 2, 3, rng.randint(4, 20)])
    sgs = rng.random() < 0.7
    prec = "mixed" if kind == "mixed" else "fp64"
    if kind == "ensemble":
        prec = rng.choice(["fp64", "mixed"])
        return _case(None, "ensemble", 32, rng.randint(4, 5), eps, rng.randint(3, 6), prec=prec, m=m, sgs=True,
                     members=rng.randint(5, 40), jmin=2, re=re)
    top = {"fp64": 11, "mixed": 12, "rosenbrock": 9, "scalar": 10, "exner": 10, "snapshot": 11}[kind]
    k = rng.randint(7, top)
    n0 = 1 << rng.randint(3, 5)
    J = k - n0.bit_length() + 1
    steps = rng.randint(1, 3) if kind == "rosenbrock" else rng.randint(4, 16)
    kw = {"prec": prec, "m": m, "order": order, "sgs": sgs, "vortices": nv, "re": re}
    if kind == "rosenbrock":
        return _case(None, "steps", n0, J, eps, steps, **dict(kw, scheme="rosenbrock"))
    if kind == "exner":
        return _case(None, "exner", n0, J, eps, steps, **dict(kw, sgs=False, scheme=rng.choice(["frozen", "rosenbrock"])))
    if kind in ("scalar", "snapshot"):
        return _case(None, kind, n0, J, eps, 0 if kind == "snapshot" else steps, **kw)
    return _case(None, "steps", n0, J, eps, steps, **kw)


# ---- inputs -------------------------------------------------------------------

def _vortices(n, rng):
    """Centres, circulations and core sizes of n Gaussian vortices."""
    if n == 2:      # the equal pair, centres jittered
        j = rng.uniform(-0.01, 0.01, (2, 2))
        return np.array([-0.6, 0.6]) + j[0], j[1].copy(), np.ones(2), np.full(2, 0.3)
    if n == 3:      # three vortices of one sign, pair distances in [1.0, 1.6]
        while True:
            r, th = 1.2 * np.sqrt(rng.uniform(0, 1, 3)), rng.uniform(0, 2 * np.pi, 3)
            x, y = r * np.cos(th), r * np.sin(th)
            if all(1.0 <= math.hypot(x[a] - x[b], y[a] - y[b]) <= 1.6 for a, b in ((0, 1), (0, 2), (1, 2))):
                return x, y, rng.uniform(0.8, 1.2, 3), np.full(3, 0.25)
    return rng.uniform(-2, 2, n), rng.uniform(-2, 2, n), rng.uniform(-1.2, 1.2, n), rng.uniform(0.2, 0.5, n)


def _runs(case, seed):
    """The parameters and vortices of the case's runs (one, or an ensemble's members)."""
    rng = np.random.default_rng(seed)
    out = []
    for q in range(case["members"]):
        p = RunParams(n0=case["n0"], J=case["J"], eps=case["eps"], re=case["re"], m=case["m"],
                      sgs=SGS_DYNAMIC if case["sgs"] else SGS_OFF, cs=CS if case["sgs"] else 0.0,
                      prec=1 if case["prec"] == "mixed" else 0, p=case["order"] // 2,
                      scheme=ROSENBROCK if case["scheme"] == "rosenbrock" else 0)
        v = _vortices(case["vortices"], rng)
        if case["kind"] == "exner":
            p.model, p.cpt, p.coriolis = EXNER, 25.0, 0.5
        if case["kind"] == "ensemble":      # levels dealt out evenly, so that the work does not hang on the seed
            p.J = case["jmin"] + q % (case["J"] - case["jmin"] + 1)
            d = rng.uniform(0.8, 2.0)
            p.re = float(rng.uniform(5000.0, 37440.0))
            v = (np.array([-0.5 * d, 0.5 * d]), np.zeros(2), np.array([1.0, rng.uniform(0.5, 1.0)]), np.full(2, 0.3))
        out.append((p, v))
    return out


def _front(NJ, seed):
    """The water-vapour front of the paper's section on vapour transport: 1 for y > 0, else 0, here
    along a gentle wave whose phase hangs on the seed."""
    x = -math.pi + 2 * math.pi / NJ * torch.arange(NJ, dtype=torch.float64, device="cuda")
    ph = float(np.random.default_rng(seed + 77).uniform(0, 2 * np.pi))
    return (x[:, None] > 0.2 * torch.sin(x + ph)[None, :]).double().contiguous()


def _field(NJ, v):
    """The sampled sum of Gaussian vortices, minimum-image distances on [-pi, pi)^2."""
    x = -math.pi + 2 * math.pi / NJ * torch.arange(NJ, dtype=torch.float64, device="cuda")
    om = torch.zeros(NJ, NJ, dtype=torch.float64, device="cuda")
    for xc, yc, g, s in zip(*v):
        dx = torch.remainder(x - xc + math.pi, 2 * math.pi) - math.pi
        dy = torch.remainder(x - yc + math.pi, 2 * math.pi) - math.pi
        om += g / (math.pi * s * s) * torch.exp(-(dx * dx)[None, :] / (s * s) - (dy * dy)[:, None] / (s * s))
    return om


class _State:
    """A run or an ensemble with the buffers its results are read into."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.stream = torch.cuda.Stream()
        self.run = self.ens = None
        self.runs = _runs(case, seed)
        cfgs = [wrc.make_config(p) for p, _ in self.runs]
        if case["kind"] == "ensemble":
            self.ens = wrc.wrc_ensemble_create(cfgs, self.stream.cuda_stream)
            self.handles = [wrc.wrc_ensemble_member(self.ens, q) for q in range(len(cfgs))]
            for h, (_, v) in zip(self.handles, self.runs):
                wrc.wrc_init_vortices(h, *v)
            wrc.wrc_ensemble_tune(self.ens, 2)
        else:
            self.run = wrc.wrc_create(cfgs[0], self.stream.cuda_stream)
            self.handles = [self.run]
        sizes = [p.NJ * p.NJ for p, _ in self.runs]
        self.at = [0] + np.cumsum(sizes).tolist()
        n = self.at[-1]
        self.val = torch.zeros(n, dtype=torch.float64, device="cuda")
        self.idx = torch.zeros(n if case["prec"] == "fp64" else 1, dtype=torch.int32, device="cuda")
        NJ = self.runs[0][0].NJ
        if case["kind"] == "scalar":
            self.front = _front(NJ, seed)
        if case["kind"] in ("scalar", "exner"):
            self.more = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2)]
        if case["kind"] == "snapshot":
            self.omega = _field(NJ, self.runs[0][1])
            self.more = [torch.zeros(NJ, NJ, dtype=torch.float64, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()

    def __del__(self):
        if getattr(self, "run", None):
            wrc.wrc_destroy(self.run)
        if getattr(self, "ens", None):
            wrc.wrc_ensemble_destroy(self.ens)


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    c = state.case
    p, v = state.runs[0]
    h, kind = state.run, c["kind"]
    if kind == "snapshot":
        wrc.wrc_init_field(h, state.omega)
        wrc.wrc_query_active(h, state.idx, state.val, state.val.numel())
        for which, out in zip((wrc.FIELD_OMEGA, wrc.FIELD_PSI, wrc.FIELD_U, wrc.FIELD_V), state.more):
            wrc.wrc_query_field(h, which, out)
        return {"idx": state.idx, "omega": state.val, **{k: f for k, f in zip(("R", "psi", "U", "V"), state.more)}}
    if kind == "exner":
        wrc.wrc_exner_init_vortices(h, *v, 1.0)
        wrc.wrc_step(h, c["steps"])
        wrc.wrc_query_exner(h, state.idx, state.val, state.more[0], state.more[1], state.val.numel())
        return {"idx": state.idx, "u": state.val, "v": state.more[0], "pi": state.more[1]}
    for hh, (_, vv) in zip(state.handles, state.runs):
        wrc.wrc_init_vortices(hh, *vv)
    if kind == "scalar":
        wrc.wrc_scalar_init(h, 1.0 / p.re, state.front)
    if state.ens:
        wrc.wrc_ensemble_step(state.ens, c["steps"])
    else:
        wrc.wrc_step(h, c["steps"])
    if c["prec"] == "mixed":
        for q, hh in enumerate(state.handles):
            wrc.wrc_query_field(hh, wrc.FIELD_OMEGA, state.val[state.at[q]:state.at[q + 1]])
        return {"R": state.val.float()}
    for q, hh in enumerate(state.handles):
        at = slice(state.at[q], state.at[q + 1])
        wrc.wrc_query_active(hh, state.idx[at], state.val[at], state.at[q + 1] - state.at[q])
    out = {"idx": state.idx, "omega": state.val}
    if kind == "scalar":
        wrc.wrc_query_scalar(h, None, state.more[0], state.more[0].numel())
        out["r_v"] = state.more[0]
    return out


# ---- what a pass cannot do without ---------------------------------------------

def _active(case, J):
    """Rough active count of a run: the coarsest points, and per vortex a count that grows as
    eps^(-1/order), limited by the lattice."""
    if case["kind"] == "scalar":
        return 60000 * (1 << J) * case["n0"] // 1024
    per = {4: 7800.0, 6: 3400.0, 8: 2700.0}[case["order"]]
    nv = min(case["vortices"], 10)
    fields = 0.5 if case["kind"] == "exner" else 1.0
    n = case["n0"] ** 2 + nv * per * fields * (1e-4 / case["eps"]) ** (2.0 / case["order"])
    return int(min(n, (case["n0"] << J) ** 2 / 4))


def work(case):
    """Bytes: the sampled field in (snapshot), the active set or the lattice out.  Operations, per step:
    the real 2-D transforms of the Poisson solve (5 N log2 N for both ways), m + 1 operator
    applications (30 operations a point), the dots and updates of one orthogonalisation against j
    vectors at Arnoldi step j (4 (j + 1) a point), the combination (2 m)."""
    by = fl = 0.0
    m = case["m"]
    for q in range(case["members"]):
        J = case["J"]
        if case["kind"] == "ensemble":
            J = case["jmin"] + q % (case["J"] - case["jmin"] + 1)
        N = float((case["n0"] << J) ** 2)
        na = _active(case, J)
        fft = 5.0 * N * math.log2(N)
        if case["kind"] == "snapshot":
            by += 8.0 * N * 5 + 12.0 * na
            fl += fft + 30.0 * N
            continue
        by += 4.0 * N if case["prec"] == "mixed" else 12.0 * na
        fields = {"exner": 3, "scalar": 2}.get(case["kind"], 1)
        by += 8.0 * na * (fields - 1) + (8.0 * N if case["kind"] == "scalar" else 0.0)
        solves = 0 if case["kind"] == "exner" else m + 1 if case["scheme"] == "rosenbrock" else 1
        kry = 30.0 * (m + 1) + sum(4.0 * (j + 1) for j in range(m)) + 2.0 * m
        fl += case["steps"] * (solves * fft + fields * na * kry)
    return {"bytes": by, "flops": fl}


# ---- the same method in plain torch, 64 bits ------------------------------------

_PRED = {2: ([9.0, -1.0], 4), 3: ([150.0, -25.0, 3.0], 8), 4: ([1225.0, -245.0, 49.0, -5.0], 11)}
_D1 = {2: ([8.0, -1.0], 12.0), 3: ([6528.0, -1272.0, 128.0, 3.0], 8760.0),
       4: ([4715520.0, -1141695.0, 199680.0, -13225.0, -1024.0, 5.0], 5946360.0)}
_D2 = {2: ([-30.0, 16.0, -1.0], 12.0), 3: ([-490.0, 270.0, -27.0, 2.0], 180.0),
       4: ([-14350.0, 8064.0, -1008.0, 128.0, -9.0], 5040.0)}


def _sh(F, axis, r):
    return torch.roll(F, -r, dims=1 if axis == 0 else 0)


class _Plain:
    """One run over dense NJ x NJ lattices [k, i] (axis 0 = x = columns)."""

    def __init__(self, p):
        self.p, self.P, self.J, self.NJ = p, p.p, p.J, p.NJ
        self.h = 2 * math.pi / p.NJ
        i = torch.arange(self.NJ, device="cuda")
        t = torch.zeros_like(i)
        for b in range(1, self.J + 1):
            t[i % (1 << b) == 0] = b
        self.lev = self.J - torch.minimum(t[:, None], t[None, :])

    # transform -----------------------------------------------------------------
    def line(self, F, axis):
        c, q = _PRED[self.P]
        acc = sum(ck * (_sh(F, axis, -(2 * k + 1)) + _sh(F, axis, 2 * k + 1)) for k, ck in enumerate(c))
        return acc * 2.0 ** -q

    def predict(self, F, j):
        s = 1 << (self.J - j)
        sub = F[::s, ::s]
        odd = torch.arange(sub.shape[0], device="cuda") % 2 == 1
        oi, ok = odd[None, :], odd[:, None]
        px = self.line(sub, 0)
        return sub, oi | ok, torch.where(oi & ~ok, px, torch.where(ok & ~oi, self.line(sub, 1), self.line(px, 1)))

    def rec(self, values, A):
        R = torch.where(A, values, torch.zeros_like(values))
        for j in range(1, self.J + 1):
            sub, new, P = self.predict(R, j)
            s = 1 << (self.J - j)
            sub.copy_(torch.where(new & ~A[::s, ::s], P, sub))
        return R

    def significant(self, R, A):
        S = self.lev == 0
        for j in range(1, self.J + 1):
            s = 1 << (self.J - j)
            sub, new, P = self.predict(R, j)
            S[::s, ::s] |= new & A[::s, ::s] & ((sub - P).abs() >= self.p.eps)
        return S

    def marks(self, src):
        odd = torch.arange(src.shape[0], device="cuda") % 2 == 1
        oi, ok = odd[None, :], odd[:, None]
        X, Y, XY = src & oi & ~ok, src & ok & ~oi, src & oi & ok
        M = torch.zeros_like(src)
        offs = [o for k in range(self.P) for o in (-(2 * k + 1), 2 * k + 1)]
        for a in offs:
            M |= _sh(X, 0, a) | _sh(Y, 1, a)
            t = _sh(XY, 0, a)
            for b in offs:
                M |= _sh(t, 1, b)
        return M

    def grid(self, S):
        A = S.clone()
        for j in range(1, self.J + 1):
            Sj = S & (self.lev == j)
            s = 1 << (self.J - j)
            st = s // 2 if j < self.J else s
            target = (self.lev == j) | (self.lev == j + 1)
            for a in range(-s, s + 1, st):
                t = _sh(Sj, 0, a)
                for b in range(-s, s + 1, st):
                    A |= _sh(t, 1, b) & target
        for j in range(self.J, 0, -1):
            s = 1 << (self.J - j)
            sub = A[::s, ::s]
            odd = torch.arange(sub.shape[0], device="cuda") % 2 == 1
            sub |= self.marks(sub & (odd[None, :] | odd[:, None]))
        return A

    def adapt(self, A, fields, whole=None):
        """The new grid and the fields' values on it; whole: per field, sampled on every point."""
        whole = whole or [False] * len(fields)
        Rs = [f if w else self.rec(f, A) for f, w in zip(fields, whole)]
        S = torch.zeros_like(self.lev, dtype=torch.bool)
        for R, w in zip(Rs, whole):
            S |= self.significant(R, torch.ones_like(S) if w else A)
        return self.grid(S), Rs

    # derivatives ----------------------------------------------------------------
    def d1(self, F, axis, h):
        n, d = _D1[self.P]
        return sum(c * (_sh(F, axis, j + 1) - _sh(F, axis, -j - 1)) for j, c in enumerate(n)) / (d * h)

    def d2(self, F, axis, h):
        n, d = _D2[self.P]
        return (n[0] * F + sum(c * (_sh(F, axis, j + 1) + _sh(F, axis, -j - 1)) for j, c in enumerate(n[1:]))) / (d * h * h)

    def freeze_grid(self, A):
        self.A = A
        self.js = []
        for axis in (0, 1):
            jj = torch.where(A, self.lev, -1)
            for j in range(self.J + 1):
                s = 1 << (self.J - j)
                sA = A[::s, ::s]
                v = jj[::s, ::s]
                v[sA & (_sh(sA, axis, 1) | _sh(sA, axis, -1))] = j
            self.js.append(jj)

    def derivs(self, q):
        """Dx, Dy, Dxx + Dyy at the active points of a compact vector q."""
        Q = torch.zeros(self.NJ, self.NJ, dtype=torch.float64, device="cuda")
        Q[self.A] = q
        R = self.rec(Q, self.A)
        out = []
        for axis in (0, 1):
            D, DD = torch.zeros_like(R), torch.zeros_like(R)
            for j in range(self.J + 1):
                s = 1 << (self.J - j)
                at = self.js[axis][::s, ::s] == j
                sub = R[::s, ::s]
                D[::s, ::s] = torch.where(at, self.d1(sub, axis, self.h * s), D[::s, ::s])
                DD[::s, ::s] = torch.where(at, self.d2(sub, axis, self.h * s), DD[::s, ::s])
            out.append((D[self.A], DD[self.A]))
        return R, out[0][0], out[1][0], out[0][1] + out[1][1]

    # flow -----------------------------------------------------------------------
    def psi(self, R):
        t = torch.arange(self.NJ, dtype=torch.float64, device="cuda") * (math.pi / self.NJ)
        n, d = _D2[self.P]
        sg = 4.0 * sum(c * torch.sin((j + 1) * t) ** 2 for j, c in enumerate(n[1:])) / (d * self.h * self.h)
        den = sg[:, None] + sg[None, :self.NJ // 2 + 1]
        den[0, 0] = 1.0
        F = torch.fft.rfft2(R) / den
        F[0, 0] = 0.0
        return torch.fft.irfft2(F, s=(self.NJ, self.NJ))

    def velocity(self, psi):
        return self.d1(psi, 1, self.h), -self.d1(psi, 0, self.h)

    def forcing(self, psi, U):
        if not self.p.sgs:
            return torch.zeros_like(psi)
        h = self.h
        S11, S12 = self.d1(U, 0, h), 0.5 * (self.d2(psi, 1, h) - self.d2(psi, 0, h))
        nut = (self.p.cs * h) ** 2 * 2.0 * torch.sqrt(S11 * S11 + S12 * S12)
        a, c = 2.0 * nut * S12, nut * S11
        return self.d2(a, 0, h) - self.d2(a, 1, h) - 4.0 * self.d1(self.d1(c, 1, h), 0, h)

    # Krylov ---------------------------------------------------------------------
    def increment(self, op, b):
        m, beta = self.p.m, torch.linalg.norm(b)
        if float(beta) == 0.0:
            return torch.zeros_like(b)
        V = torch.zeros(m + 1, b.numel(), dtype=torch.float64, device="cuda")
        H = torch.zeros(m + 1, m, dtype=torch.float64, device="cuda")
        V[0], k = b / beta, m
        for j in range(m):
            w = op(V[j])
            wn = torch.linalg.norm(w)
            for _ in range(2):
                c = V[:j + 1] @ w
                w = w - c @ V[:j + 1]
                H[:j + 1, j] += c
            H[j + 1, j] = torch.linalg.norm(w)
            if float(H[j + 1, j]) <= 1e-12 * float(wn):
                k = j + 1
                break
            V[j + 1] = w / H[j + 1, j]
        M = torch.zeros(k + 1, k + 1, dtype=torch.float64)
        M[:k, :k] = self.p.dt * H[:k, :k].cpu()
        M[0, k] = 1.0
        y = torch.linalg.matrix_exp(M)[:k, k].cuda()
        return self.p.dt * beta * (y @ V[:k])

    def step(self, A, om, rv=None):
        """One vorticity step on (A, om); with a scalar also rv.  Lattice arrays."""
        p = self.p
        self.freeze_grid(A)
        R, wx, wy, wl = self.derivs(om[A])
        psi = self.psi(R)
        U, V = self.velocity(psi)
        g = self.forcing(psi, U)[A]
        U, V = U[A], V[A]
        nu = 1.0 / p.re

        def op(q, nu=nu):
            Q, x, y, lap = self.derivs(q)
            w = -U * x - V * y + nu * lap
            if p.scheme == ROSENBROCK:
                u2, v2 = self.velocity(self.psi(Q))
                w = w - u2[A] * wx - v2[A] * wy
            return w

        fields = [om]
        inc = [self.increment(op, -U * wx - V * wy + nu * wl + g)]
        if rv is not None:
            _, x, y, lap = self.derivs(rv[A])
            fields.append(rv)
            inc.append(self.increment(op, -U * x - V * y + nu * lap))
        new = []
        for f, d in zip(fields, inc):
            n = f.clone()
            n[A] = f[A] + d
            new.append(n)
        return self.adapt(A, new)

    def exner_step(self, A, f):
        p = self.p
        self.freeze_grid(A)
        u, v, q = (x[A] for x in f)
        (_, ux, uy, ul), (_, vx, vy, vl), (_, qx, qy, _) = self.derivs(u), self.derivs(v), self.derivs(q)
        C, co, nu = p.cpt, p.coriolis, 1.0 / p.re

        def op(x):
            du, dv, dq = x.chunk(3)
            (_, dux, duy, dul), (_, dvx, dvy, dvl), (_, dqx, dqy, _) = self.derivs(du), self.derivs(dv), self.derivs(dq)
            a = -(u * dux + v * duy) - C * dqx + co * dv + nu * dul
            b = -(u * dvx + v * dvy) - C * dqy - co * du + nu * dvl
            c = -(u * dqx + v * dqy) - q * (dux + dvy)
            if p.scheme == ROSENBROCK:
                a = a - (du * ux + dv * uy)
                b = b - (du * vx + dv * vy)
                c = c - (du * qx + dv * qy) - dq * (ux + vy)
            return torch.cat([a, b, c])

        rhs = torch.cat([-(u * ux + v * uy) - C * qx + co * v + nu * ul, -(u * vx + v * vy) - C * qy - co * u + nu * vl,
                         -(u * qx + v * qy) - q * (ux + vy)])
        new = []
        for x, d in zip(f, self.increment(op, rhs).chunk(3)):
            n = x.clone()
            n[A] = x[A] + d
            new.append(n)
        return self.adapt(A, new)


def _at(f, A):
    """The active values, in order, followed by zeros: a result buffer."""
    x = torch.zeros(f.numel(), dtype=torch.float64, device="cuda")
    v = f[A]
    x[:v.numel()] = v
    return x


def exact(case, seed):
    if case["kind"] == "ensemble" and case["members"] * case["steps"] > 110:
        return None      # over 20 seconds
    out = []
    for p, v in _runs(case, seed):
        S = _Plain(p)
        full = torch.ones(p.NJ, p.NJ, dtype=torch.bool, device="cuda")
        om = _field(p.NJ, v)
        if case["kind"] == "exner":
            u, w = S.velocity(S.psi(om))
            A, f = S.adapt(full, [u, w, torch.ones_like(u)], [True] * 3)
            for _ in range(case["steps"]):
                A, f = S.exner_step(A, f)
            return {"idx": None, "u": _at(f[0], A), "v": _at(f[1], A), "pi": _at(f[2], A)}
        A, f = S.adapt(full, [om], [True])
        if case["kind"] == "snapshot":
            R = S.rec(f[0], A)
            psi = S.psi(R)
            U, V = S.velocity(psi)
            return {"idx": None, "omega": _at(f[0], A), "R": R, "psi": psi, "U": U, "V": V}
        if case["kind"] == "scalar":
            A, f = S.adapt(A, [f[0], _front(p.NJ, seed)], [False, True])
        for _ in range(case["steps"]):
            A, f = S.step(A, *f)
        if case["kind"] == "scalar":
            return {"idx": None, "omega": _at(f[0], A), "r_v": _at(f[1], A)}
        out.append(S.rec(f[0], A).reshape(-1) if case["prec"] == "mixed" else _at(f[0], A))
    x = torch.cat(out)
    return {"R": x} if case["prec"] == "mixed" else {"idx": None, "omega": x}
