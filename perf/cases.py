"""The work that users of the solver have it do, as measured cases: whole runs, single stage operators,
vector-Jacobian products, gradients, batches and block decompositions, over the range of meshes, fluxes,
boundary conditions and time schemes in use.

``prepare`` makes the inputs and the handle a program keeps; ``run`` is one pass through the public
entry points; ``exact`` evaluates the same scheme in plain torch float64 (class ``_Scheme``, written from
the paper's formulas in their textbook form: full moments, 4x4 projections, autograd for derivatives).
"""
import math

import numpy as np
import torch

from paper_2402_10914_gb300 import solver as S
from paper_2402_10914_gb300.inputs import GKS, LF, OUTFLOW, PERIODIC, REFLECT, S2O4, SSPRK3, Settings

_BC = {"periodic": (PERIODIC,) * 4, "outflow": (OUTFLOW,) * 4, "reflect": (REFLECT,) * 4,
       "strip": (OUTFLOW, OUTFLOW, PERIODIC, PERIODIC)}
_SIDES = (64, 96, 128, 192, 256, 384, 512)


def _case(name, kind, init, nx, ny, bc, flux, steps=1, scheme="s2o4", limiter=True, **more):
    case = dict(kind=kind, init=init, nx=nx, ny=ny, bc=bc, flux=flux, steps=steps, scheme=scheme, limiter=limiter, **more)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the paper's one-dimensional problems run as a strip of four rows: the smallest calls, all latency
        _case("strip_gks_100x4", "run", "strip", 100, 4, "strip", "gks", steps=8),
        # the accuracy study's density wave: a whole 20-step L-F run on a small periodic mesh
        _case("wave_lf_40x40", "run", "wave", 40, 40, "periodic", "lf", steps=20, limiter=False),
        # one stage operator on an odd mesh, as a caller with an own time integrator asks for it
        _case("stage_gks_97x61", "stage", "smooth", 97, 61, "periodic", "gks"),
        # the benchmark's four-quadrant Riemann problem at its own size
        _case("quadrants_gks_400x400", "run", "quadrants", 400, 400, "outflow", "gks", steps=4),
        # the paper's pairing of L-F with SSP-RK3 on a rectangular mesh with odd sides
        _case("quadrants_lf_rk3_333x217", "run", "quadrants", 333, 217, "outflow", "lf", steps=4, scheme="ssprk3"),
        # the robustness run's largest mesh, walls all round, pressure ratio 1e6
        _case("blast_gks_2048x2048", "run", "blast", 2048, 2048, "reflect", "gks", steps=1),
        # one stage operator on a large ragged mesh
        _case("stage_gks_1021x509", "stage", "quadrants", 1021, 509, "outflow", "gks"),
        # training: the gradient of a final-time functional through the checkpointed run (autograd).  Derivatives
        # are compared on smooth data, and on larger meshes without the time limiter: at a kink of the scheme
        # (|p_l - p_r| in uniform pressure, a tie in the limiter's minimum) they follow the last bit of the state
        _case("gradient_gks_256x256", "gradient", "smooth", 256, 256, "periodic", "gks", steps=10, limiter=False, every=5),
        # reverse of a single stage operator, for callers that differentiate their own integrator
        _case("vjp_gks_67x83", "vjp", "smooth", 67, 83, "periodic", "gks"),
        _case("vjp_lf_400x400", "vjp", "wave", 400, 400, "periodic", "lf", limiter=False),
        # serving: independent problems of uneven sizes and mixed fluxes advanced in one graph launch
        _case("batch_16_mixed", "batch", "quadrants", 0, 0, "outflow", "mixed", steps=4, count=16, sides=1000),
        # one mesh split in 3 x 2 blocks with halo exchange
        _case("blocks_gks_300x200", "blocks", "smooth", 300, 200, "periodic", "gks", steps=4, px=3, py=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("run", "run", "run", "stage", "stage", "vjp", "gradient", "batch", "blocks"))
    flux = rng.choice(("gks", "gks", "lf"))
    init, bc = rng.choice((("wave", "periodic"), ("smooth", "periodic"), ("quadrants", "outflow"), ("vortex", "periodic"),
                           ("blast", "reflect"), ("strip", "strip")))
    if kind in ("vjp", "gradient") or (init in ("blast", "strip") and kind != "run"):
        init, bc = "smooth", "periodic"
    limiter = kind not in ("vjp", "gradient") and init != "wave"
    if kind == "gradient":
        return _case("", kind, init, _log_int(rng, 24, 256), _log_int(rng, 24, 256), bc, flux, steps=rng.randint(2, 10),
                     limiter=limiter, every=rng.randint(2, 5))
    if kind == "batch":
        return _case("", kind, "quadrants", 0, 0, "outflow", "mixed", steps=rng.randint(1, 5), count=rng.randint(3, 16),
                     sides=rng.randint(1, 1 << 20))
    if init == "strip":
        nx, ny = _log_int(rng, 50, 400), 4
    elif init == "blast":
        nx = ny = _log_int(rng, 128, 1600)
    elif kind == "blocks":
        nx, ny = _log_int(rng, 40, 400), _log_int(rng, 40, 400)
    elif kind == "vjp":
        nx, ny = _log_int(rng, 24, 500), _log_int(rng, 24, 500)
    else:
        nx, ny = _log_int(rng, 24, 1100), _log_int(rng, 24, 1100)
    steps = max(1, min(10, int(2.0e6 / (nx * ny)))) if kind in ("run", "blocks") and init != "blast" else 1
    more = dict(px=rng.randint(1, 4), py=rng.randint(1, 3)) if kind == "blocks" else {}
    return _case("", kind, init, nx, ny, bc, flux, steps=steps, limiter=limiter,
                 scheme="ssprk3" if kind == "run" and flux == "lf" and rng.random() < 0.6 else "s2o4", **more)


# ---------------------------------------------------------------------------------------------------
# settings and inputs
# ---------------------------------------------------------------------------------------------------
_BOX = {"strip": (0.0, 1.0), "wave": (0.0, 2.0), "smooth": (0.0, 1.0), "quadrants": (0.0, 1.0), "vortex": (0.0, 10.0),
        "blast": (0.0, 1.0)}


def _settings(case, nx, ny, flux):
    init = case["init"]
    lo, hi = _BOX[init]
    y1 = lo + (hi - lo) * ny / nx if init == "strip" else hi
    return Settings(nx=nx, ny=ny, x0=lo, x1=hi, y0=lo, y1=y1, cfl=0.4 if init == "blast" else 0.5, bc=_BC[case["bc"]],
                    flux=GKS if flux == "gks" else LF, time_limiter=int(case["limiter"]),
                    time_scheme=SSPRK3 if case["scheme"] == "ssprk3" else S2O4)


def _field(init, s, seed):
    """Conserved cell averages [4][ny][nx] of a seeded initial state (host, float64)."""
    rng = np.random.default_rng(seed)
    dx, dy = (s.x1 - s.x0) / s.nx, (s.y1 - s.y0) / s.ny
    X, Y = np.meshgrid(s.x0 + (np.arange(s.nx) + 0.5) * dx, s.y0 + (np.arange(s.ny) + 0.5) * dy)
    one = np.ones_like(X)

    def wave(amp):                      # a few low Fourier modes that close on the box
        f = np.zeros_like(X)
        for _ in range(3):
            kx, ky = rng.integers(1, 3, size=2)
            f += rng.uniform(-1, 1) * np.sin(2 * np.pi * (kx * (X - s.x0) / (s.x1 - s.x0) + ky * (Y - s.y0) / (s.y1 - s.y0))
                                             + rng.uniform(0, 2 * np.pi))
        return amp * f

    if init == "wave":                  # rho = 1 + a sin(pi (x + y) + phase), u = v = p = 1
        rho = 1.0 + rng.uniform(0.1, 0.25) * np.sin(np.pi * (X + Y) + rng.uniform(0, 2 * np.pi))
        u, v, p = one, one, one
    elif init == "smooth":
        rho, u, v, p = 1.0 + wave(0.1), 0.3 + wave(0.1), -0.2 + wave(0.1), 1.0 + wave(0.1)
    elif init == "vortex":              # isentropic vortex of strength 5 in a unit background, noisy density; its
        cx, cy = rng.uniform(4.5, 5.5, 2)   # centre is off the mesh lines, where mirror symmetry ties branches
        r2 = (X - cx) ** 2 + (Y - cy) ** 2
        f = 5.0 / (2 * np.pi) * np.exp(0.5 * (1.0 - r2))
        u, v = 1.0 - f * (Y - cy), 1.0 + f * (X - cx)
        T = 1.0 - 0.4 * 25.0 / (8 * 1.4 * np.pi ** 2) * np.exp(1.0 - r2)
        rho = T ** 2.5
        p = rho * T
        rho = rho + rng.normal(0.0, 1e-3, X.shape)
    elif init == "quadrants":           # four random states split at the centre, with a weak smooth wave on top
        q = np.where(Y < 0.5, np.where(X < 0.5, 0, 1), np.where(X >= 0.5, 2, 3))
        st = np.stack([rng.uniform(0.2, 2.0, 4), rng.uniform(-0.75, 0.75, 4), rng.uniform(-0.75, 0.75, 4), rng.uniform(0.2, 2.0, 4)])
        rho, u, v, p = (st[k][q] * (1.0 + wave(0.01)) for k in range(4))
    elif init == "blast":               # pressure ratio 1e6 inside a disc, with density noise
        r = rng.uniform(0.09, 0.11)
        p = np.where((X - 0.5) ** 2 + (Y - 0.5) ** 2 < r * r, 1e4, 0.01)
        rho, u, v = 1.0 + rng.normal(0.0, 1e-3, X.shape), 0.0 * one, 0.0 * one
    else:                               # strip: two receding streams (123 problem) of moderate Mach number
        m = rng.uniform(0.8, 1.5)
        u = np.where(X < 0.5, -2.0, 2.0)
        rho, v, p = 1.0 + 0.01 * np.sin(2 * np.pi * X + rng.uniform(0, 6)), 0.0 * one, 4.0 / (1.4 * m * m) * one
    return np.stack([rho, rho * u, rho * v, p / (s.gamma - 1.0) + 0.5 * rho * (u * u + v * v)])


def _alpha(s, seed):
    """A DF field as a run leaves it: one in smooth flow, scattered below the threshold in a patch."""
    rng = np.random.default_rng(seed + 77)
    a = np.ones((s.ny, s.nx))
    h, w = max(1, s.ny // 8), max(1, s.nx // 8)
    a[:h, :w] = rng.uniform(0.0, 1.0, (h, w))
    return a


def _members(case):
    """Side and flux of each problem of a batch, from the case alone."""
    rng = np.random.default_rng(case["sides"])
    return [(int(rng.choice(_SIDES)), "gks" if rng.uniform() < 0.5 else "lf") for _ in range(case["count"])]


def _stage_dt(s):
    return 0.2 * min((s.x1 - s.x0) / s.nx, (s.y1 - s.y0) / s.ny) / 3.0


def _inputs(case, seed):
    """Everything numeric a case starts from, on the host."""
    if case["kind"] == "batch":
        sets = [_settings(case, n, n, f) for n, f in _members(case)]
        return sets, [_field(case["init"], s, 1000 * seed + k) for k, s in enumerate(sets)]
    s = _settings(case, case["nx"], case["ny"], case["flux"])
    d = {"W": _field(case["init"], s, seed)}
    if case["kind"] in ("stage", "vjp"):
        d["alpha"] = _alpha(s, seed)
    if case["kind"] == "vjp":
        rng = np.random.default_rng(seed + 5)
        dt = _stage_dt(s)
        d["bars"] = [rng.normal(size=d["W"].shape), dt * rng.normal(size=d["W"].shape), dt * rng.normal(size=d["W"].shape)]
    if case["kind"] == "gradient":
        d["bar"] = np.random.default_rng(seed + 5).normal(size=d["W"].shape)
    return s, d


def _cuda(a):
    return torch.as_tensor(a, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    s, d = _inputs(case, seed)
    st = {"case": case, "s": s}
    if case["kind"] == "batch":
        st["solver"] = S.BatchSolver(s)
        st["W"] = d
        st["solver"].prepare(case["steps"])
        return st
    if case["kind"] == "blocks":
        st["solver"] = S.DecompSolver(s, case["px"], case["py"])
        st["W"] = d["W"]
        return st
    st["solver"] = S.Solver(s)
    st.update({k: [_cuda(b) for b in v] if isinstance(v, list) else _cuda(v) for k, v in d.items()})
    return st


def run(st):
    case, sol = st["case"], st["solver"]
    kind = case["kind"]
    if kind == "run":                      # load a state, advance it, read the result on the device
        sol.set_ic(st["W"])
        sol.step(case["steps"])
        W, a, t, n = sol.get_state(device=True)
        return {"W": W, "alpha": a, "t": t, "step": n}
    if kind == "stage":
        return list(sol.residual(st["W"], st["alpha"], _stage_dt(st["s"])))
    if kind == "vjp":
        return S.adjoint_residual(sol, st["W"], st["alpha"], _stage_dt(st["s"]), *st["bars"])
    if kind == "gradient":
        W0 = st["W"].clone().requires_grad_(True)
        W = S.GKSRun.apply(W0, sol, case["steps"], case["every"])
        W.backward(st["bar"])
        return {"W": W.detach(), "gradient": W0.grad}
    if kind == "batch":
        for p, W in enumerate(st["W"]):
            sol.set_ic(p, W)
        sol.step(case["steps"])
        return [sol.get_state(p)[:2] for p in range(case["count"])]
    sol.set_ic(st["W"])                     # blocks
    sol.step(case["steps"])
    W, a, t, n = sol.get_state()
    return {"W": W, "alpha": a, "t": t, "step": n}


# FP64 operations that the scheme's formulas need per face line (two normal reconstructions of four
# characteristic variables), face side (four tangential ones) and Gauss point (flux and its time derivative)
_LINE, _SIDE, _POINT = 1000.0, 540.0, {"gks": 850.0, "lf": 250.0}


def _stage_flops(nx, ny, flux):
    faces, lines = (nx + 1) * ny + nx * (ny + 1), (nx + 1) * (ny + 4) + (nx + 4) * (ny + 1)
    return lines * _LINE + 2 * faces * (_SIDE + _POINT[flux])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = [(a, f) for a, f in _members(case)]
        return {"bytes": float(sum(a * a * 9 * 8 for a, _ in n)),
                "flops": float(sum(2 * case["steps"] * _stage_flops(a, a, f) for a, f in n))}
    nx, ny = case["nx"], case["ny"]
    one, cells = _stage_flops(nx, ny, case["flux"]), nx * ny
    stages = {"stage": 1, "vjp": 1}.get(kind, (3 if case["scheme"] == "ssprk3" else 2) * case["steps"])
    # a reverse sweep costs about twice its forward in operations; a gradient needs one forward and one reverse
    times = 3.0 if kind in ("vjp", "gradient") else 1.0
    fields = {"stage": 5 + 13, "vjp": 5 + 12 + 4, "gradient": 4 + 4 + 8}.get(kind, 4 + 5)
    return {"bytes": float(fields * cells * 8), "flops": float(times * stages * one)}


# ---------------------------------------------------------------------------------------------------
# the scheme in plain torch float64
# ---------------------------------------------------------------------------------------------------
class _Scheme:
    """The hybrid DF + WENO-AO finite-volume scheme (arXiv 2402.10914, Sect. 2-3) on one mesh.  A sweep
    works on the x direction; the y direction is the field rotated by a quarter turn (Sect. 2.1)."""

    def __init__(self, s, device):
        self.s, self.dev = s, device
        self.dx, self.dy = (s.x1 - s.x0) / s.nx, (s.y1 - s.y0) / s.ny
        self.gm1 = s.gamma - 1.0
        self.K = (4.0 - 2.0 * s.gamma) / self.gm1
        self.d = [(1 - s.dH) * (1 - s.dL) / 2, (1 - s.dH) * s.dL, (1 - s.dH) * (1 - s.dL) / 2, s.dH]

    # -- mesh ---------------------------------------------------------------------------------
    def _map(self, n, lo, hi):
        k = torch.arange(-3, n + 3, device=self.dev)
        mirror = ((k < 0) & (lo == REFLECT)) | ((k >= n) & (hi == REFLECT))
        low = {PERIODIC: k + n, OUTFLOW: torch.zeros_like(k), REFLECT: -1 - k}[lo]
        high = {PERIODIC: k - n, OUTFLOW: torch.full_like(k, n - 1), REFLECT: 2 * n - 1 - k}[hi]
        return torch.where(k < 0, low, torch.where(k >= n, high, k)), mirror

    def pad(self, W, alpha):
        s = self.s
        ix, mx = self._map(s.nx, s.bc[0], s.bc[1])
        iy, my = self._map(s.ny, s.bc[2], s.bc[3])
        P = W[:, iy][:, :, ix]
        sx, sy = torch.where(mx, -1.0, 1.0).double(), torch.where(my, -1.0, 1.0).double()
        P = torch.stack([P[0], P[1] * sx[None, :], P[2] * sy[:, None], P[3]])
        return P, alpha[iy][:, ix]

    # -- reconstruction -----------------------------------------------------------------------
    def _basis(self, Wm):
        r, m, n, E = Wm
        u, v = m / r, n / r
        q2 = 0.5 * (u * u + v * v)
        p = self.gm1 * (E - r * q2)
        c = torch.sqrt(self.s.gamma * p / r)
        H, b1 = (E + p) / r, self.gm1 / (c * c)
        b2, z, o = q2 * b1, torch.zeros_like(u), torch.ones_like(u)
        L = [[0.5 * (b2 + u / c), 0.5 * (-b1 * u - 1 / c), -0.5 * b1 * v, 0.5 * b1],
             [1 - b2, b1 * u, b1 * v, -b1],
             [-v, z, o, z],
             [0.5 * (b2 - u / c), 0.5 * (-b1 * u + 1 / c), -0.5 * b1 * v, 0.5 * b1]]
        R = [[o, o, z, o], [u - c, u, z, u + c], [v, v, o, v], [H - u * c, q2, v, H + u * c]]
        return L, R

    @staticmethod
    def _mul(M, q):
        return [sum(M[i][k] * q[k] for k in range(4)) for i in range(4)]

    def _ao(self, q):
        """Coefficients of 1, x, x^2, x^3, x^4 (cell-centred) of the WENO-AO polynomial and its ratios r_k."""
        m2, m1, c, p1, p2 = q
        s = self.s
        subs = [(c, 0.5 * m2 - 2 * m1 + 1.5 * c, 0.5 * (m2 - 2 * m1 + c)),
                (c, 0.5 * (p1 - m1), 0.5 * (m1 - 2 * c + p1)),
                (c, -1.5 * c + 2 * p1 - 0.5 * p2, 0.5 * (c - 2 * p1 + p2))]
        a1 = (5 * (m2 - p2) - 34 * (m1 - p1)) / 48
        a2 = (-(m2 + p2) + 12 * (m1 + p1) - 22 * c) / 16
        a3 = (-(m2 - p2) + 2 * (m1 - p1)) / 12
        a4 = (m2 + p2 - 4 * (m1 + p1) + 6 * c) / 24
        beta = [b * b + 13.0 / 3.0 * e * e for _, b, e in subs]
        beta.append(a1 * a1 + a1 * a3 / 2 + 13.0 / 3.0 * a2 * a2 + 21.0 / 5.0 * a2 * a4 + 3129.0 / 80.0 * a3 * a3
                    + 87617.0 / 140.0 * a4 * a4)
        tau = ((beta[3] - beta[0]).abs() + (beta[3] - beta[1]).abs() + (beta[3] - beta[2]).abs()) / 3.0
        r = [tau / (b + s.eps) for b in beta]
        w = [self.d[k] * (1 + r[k] * r[k]) for k in range(4)]
        tot = w[0] + w[1] + w[2] + w[3]
        c3 = w[3] / tot / self.d[3]
        ck = [w[k] / tot - c3 * self.d[k] for k in range(3)] + [c3]
        A1 = sum(ck[k] * (subs[k][1] if k < 3 else a1) for k in range(4))
        A2 = sum(ck[k] * (subs[k][2] if k < 3 else a2) for k in range(4))
        return (c, A1, A2, c3 * a3, c3 * a4), r

    @staticmethod
    def _at(P, x):
        """Value and derivative of a zero-mean-corrected polynomial at x."""
        q, A1, A2, A3, A4 = P
        return (q + A1 * x + A2 * (x * x - 1 / 12) + A3 * x ** 3 + A4 * (x ** 4 - 1 / 80),
                A1 + 2 * A2 * x + 3 * A3 * x * x + 4 * A4 * x ** 3)

    @staticmethod
    def _df(q, alpha):
        _, m1, c, p1, _ = q
        return (c, alpha * 0.5 * (p1 - m1), alpha * 0.5 * (m1 - 2 * c + p1), torch.zeros_like(c), torch.zeros_like(c))

    def sweep(self, P, A, dn, dtan, dt, flux):
        """Face fluxes of one direction of a padded field: (F, dF, omega, alpha_1, alpha_2), each [nt][nn+1]."""
        s, g = self.s, math.sqrt(3.0) / 6.0
        nt, nn = P.shape[1] - 6, P.shape[2] - 6
        rows = slice(1, nt + 5)
        Wc = [[P[k, rows, f:f + nn + 1] for k in range(4)] for f in range(6)]
        al = [A[rows, f:f + nn + 1] for f in range(6)]
        Lm, Rm = self._basis([0.5 * (Wc[2][k] + Wc[3][k]) for k in range(4)])
        Q = [self._mul(Lm, w) for w in Wc]
        dfs = [torch.maximum(torch.maximum(al[1 + e], al[2 + e]), al[3 + e]) < s.alpha_thres for e in (0, 1)]
        om = torch.ones_like(al[0])
        val, slo = [[], []], [[], []]
        for k in range(4):
            for e in (0, 1):
                q = [Q[i][k] for i in range(5)] if e == 0 else [Q[5 - i][k] for i in range(5)]
                ao, r = self._ao(q)
                if s.time_limiter:
                    rr = torch.stack(r)
                    hi, lo = 1 + rr.amax(0) ** 2, 1 + rr.amin(0) ** 2
                    om = torch.minimum(om, 2 * lo / (hi + lo))
                va, sa = self._at(ao, 0.5)
                vd, sd = self._at(self._df(q, al[2 + e]), 0.5)
                val[e].append(torch.where(dfs[e], vd, va))
                slo[e].append(torch.where(dfs[e], sd, sa) * ((1 if e == 0 else -1) / dn))
        W_face = [self._mul(Rm, v) for v in val]
        W_norm = [self._mul(Rm, v) for v in slo]
        mid = slice(2, nt + 2)
        cut = lambda M: [[x[mid] for x in row] for row in M]  # noqa: E731
        L0, R0 = cut(Lm), cut(Rm)
        pts = [[None, None], [None, None]]                     # [Gauss point][side] = (W, Wn, Wt)
        for e in (0, 1):
            Ql = [self._mul(L0, [W_face[e][k][b:b + nt] for k in range(4)]) for b in range(5)]
            col = slice(2 + e, 2 + e + nn + 1)
            ac = [A[b:b + nt, col] for b in (2, 3, 4)]
            df = torch.maximum(torch.maximum(ac[0], ac[1]), ac[2]) < s.alpha_thres
            mean = [P[k, 3:3 + nt, col] for k in range(4)]
            v, d = [[], []], [[], []]
            for k in range(4):
                q = [Ql[b][k] for b in range(5)]
                ao, _ = self._ao(q)
                pd = self._df(q, ac[1])
                for m, x in enumerate((-g, g)):
                    (va, sa), (vd, sd) = self._at(ao, x), self._at(pd, x)
                    v[m].append(torch.where(df, vd, va))
                    d[m].append(torch.where(df, sd, sa) / dtan)
            for m in (0, 1):
                W, Wt, Wn = self._mul(R0, v[m]), self._mul(R0, d[m]), [x[mid] for x in W_norm[e]]
                if s.gp_fallback:
                    rp = W[0] * W[3] - 0.5 * (W[1] * W[1] + W[2] * W[2])
                    bad = ~((W[0] > 0) & (rp > 0))
                    W = [torch.where(bad, mean[k], W[k]) for k in range(4)]
                    Wn, Wt = ([torch.where(bad, torch.zeros_like(x), x) for x in y] for y in (Wn, Wt))
                pts[m][e] = (W, Wn, Wt)
        F, dF, a = [], [], []
        for m in (0, 1):
            a.append(self._alpha_point(pts[m][0][0], pts[m][1][0]).detach())
            f, d = self._gks(pts[m][0], pts[m][1], dt) if flux == GKS else self._lf(pts[m][0], pts[m][1])
            F.append(torch.stack(f))
            dF.append(torch.stack(d))
        return 0.5 * (F[0] + F[1]), 0.5 * (dF[0] + dF[1]), om[mid], a[0], a[1]

    # -- point fluxes -------------------------------------------------------------------------
    def _prim(self, W):
        u, v = W[1] / W[0], W[2] / W[0]
        return W[0], u, v, self.gm1 * (W[3] - 0.5 * W[0] * (u * u + v * v))

    def _alpha_point(self, WL, WR):
        (rl, ul, vl, pl), (rr, ur, vr, pr) = self._prim(WL), self._prim(WR)
        cl, cr = torch.sqrt(self.s.gamma * pl / rl), torch.sqrt(self.s.gamma * pr / rr)
        D = (pl - pr).abs() * (1 / pl + 1 / pr) + (ul / cl - ur / cr) ** 2 + (vl / cl - vr / cr) ** 2
        return 1 / (1 + D * D)

    def _moments(self, W, half):
        rho, U, V, p = self._prim(W)
        th = p / rho
        if half == 0:
            mu = [torch.ones_like(U), U]
        else:
            x = half * U / torch.sqrt(2 * th)
            m0 = 0.5 * torch.special.erfc(-x)
            mu = [m0, U * m0 + half * torch.sqrt(th / (2 * math.pi)) * torch.exp(-x * x)]
        mv = [torch.ones_like(V), V]
        for n in range(2, 7):
            mu.append(U * mu[-1] + (n - 1) * th * mu[-2])
            mv.append(V * mv[-1] + (n - 1) * th * mv[-2])
        mx = [torch.ones_like(V), self.K * th, self.K * (self.K + 2) * th * th]
        return mu, mv, mx

    @staticmethod
    def _psi(M, k, l, c=0):
        mu, mv, mx = M
        e = lambda a, b, x: mu[a] * mv[b] * mx[x]  # noqa: E731
        return [e(k, l, c), e(k + 1, l, c), e(k, l + 1, c), 0.5 * (e(k + 2, l, c) + e(k, l + 2, c) + e(k, l, c + 1))]

    def _apsi(self, M, a, k, l):
        p = [self._psi(M, k, l), self._psi(M, k + 1, l), self._psi(M, k, l + 1), self._psi(M, k + 2, l), self._psi(M, k, l + 2),
             self._psi(M, k, l, 1)]
        return [a[0] * p[0][i] + a[1] * p[1][i] + a[2] * p[2][i] + 0.5 * a[3] * (p[3][i] + p[4][i] + p[5][i]) for i in range(4)]

    def _slope(self, W, b):
        """a with <a psi> = b / rho for the Maxwellian of W."""
        rho, U, V, p = self._prim(W)
        lam = 0.5 * rho / p
        b = [x / rho for x in b]
        q = U * U + V * V + (self.K + 2) / (2 * lam)
        r2, r3, r4 = b[1] - U * b[0], b[2] - V * b[0], 2 * b[3] - q * b[0]
        a3 = 4 * lam * lam / (self.K + 2) * (r4 - 2 * U * r2 - 2 * V * r3)
        a2, a1 = 2 * lam * r3 - V * a3, 2 * lam * r2 - U * a3
        return [b[0] - U * a1 - V * a2 - 0.5 * a3 * q, a1, a2, a3]

    def _gks(self, left, right, dt):
        """Second-order gas-kinetic flux and time derivative (Sect. 2.2, Eqs. 25-27), zero physical collision time."""
        s = self.s
        sides = []
        for (W, Wn, Wt), half in ((left, 1), (right, -1)):
            M = self._moments(W, half)
            sides.append((W[0], M, self._slope(W, Wn), self._slope(W, Wt)))
        tot = lambda f: [sum(x) for x in zip(*[[rho * y for y in f(M, ax, ay)] for rho, M, ax, ay in sides])]  # noqa: E731
        add = lambda x, y: [a + b for a, b in zip(x, y)]  # noqa: E731
        Wc = tot(lambda M, ax, ay: self._psi(M, 0, 0))
        Mc = self._moments(Wc, 0)
        ax, ay = (self._slope(Wc, tot(lambda M, x, y, i=i: self._apsi(M, (x, y)[i], 0, 0))) for i in (0, 1))
        At = self._slope(Wc, [-Wc[0] * x for x in add(self._apsi(Mc, ax, 1, 0), self._apsi(Mc, ay, 0, 1))])
        c0, c2 = self._psi(Mc, 1, 0), self._apsi(Mc, At, 1, 0)
        c1 = add(self._apsi(Mc, ax, 2, 0), self._apsi(Mc, ay, 1, 1))
        g0 = tot(lambda M, x, y: self._psi(M, 1, 0))
        g1 = tot(lambda M, x, y: add(self._apsi(M, x, 2, 0), self._apsi(M, y, 1, 1)))
        pl, pr = self._prim(left[0])[3], self._prim(right[0])[3]
        r = s.C1 + s.C2 * ((pl - pr) / (pl + pr)).abs()
        E2 = torch.exp(-0.5 / r)
        o, T = 1 - E2, r * dt
        S3 = o * (3 - E2)
        gF, gD = r * S3, -4 * r * o * o / dt
        aF = T * T * S3 / dt - 2 * T * E2 + T * E2 * E2
        aD = 4 * (-T * T * o * o + T * dt * E2 * o) / (dt * dt)
        F, dF = [], []
        for i in range(4):
            e0, e1, e2 = Wc[0] * c0[i], Wc[0] * c1[i], Wc[0] * c2[i]
            F.append((1 - gF) * e0 + aF * e1 + gF * g0[i] - aF * g1[i])
            dF.append(-gD * e0 + aD * e1 + e2 + gD * g0[i] - aD * g1[i])
        return F, dF

    def _lf(self, left, right):
        """Lax-Friedrichs flux (Sect. 2.3) with W_t from the Euler equations and a frozen wave speed."""
        gm1, out = self.gm1, []
        for W, Wn, Wt in (left, right):
            rho, u, v, p = self._prim(W)
            q, H = 0.5 * (u * u + v * v), (W[3] + p) / W[0]

            def jac(X, n):
                dp = gm1 * (X[3] - u * X[1] - v * X[2] + q * X[0])
                w, m = ((u, X[1]), (v, X[2]))[n]
                d = m - w * X[0]
                y = [m, u * d + w * X[1], v * d + w * X[2], w * (X[3] + dp) + H * d]
                y[1 + n] = y[1 + n] + dp
                return y

            dWdt = [-(a + b) for a, b in zip(jac(Wn, 0), jac(Wt, 1))]
            flux = [W[1], W[1] * u + p, W[1] * v, u * (W[3] + p)]
            out.append((W, flux, dWdt, jac(dWdt, 0), u.abs() + torch.sqrt(self.s.gamma * p / rho)))
        (WL, FL, tL, AL, sL), (WR, FR, tR, AR, sR) = out
        c = torch.maximum(sL, sR)
        return ([0.5 * (FL[i] + FR[i]) - 0.5 * c * (WR[i] - WL[i]) for i in range(4)],
                [0.5 * (AL[i] + AR[i]) - 0.5 * c * (tR[i] - tL[i]) for i in range(4)])

    # -- stage and step -----------------------------------------------------------------------
    def stage(self, W, alpha, dt, flux=None):
        """(L, dL/dt, limited dL/dt, alpha_next) of Eq. 2."""
        flux = self.s.flux if flux is None else flux
        P, A = self.pad(W, alpha)
        F, dF, om, a1, a2 = self.sweep(P, A, self.dx, self.dy, dt, flux)
        turn = lambda x: torch.flip(x.transpose(-1, -2), (-2,))  # noqa: E731
        back = lambda x: torch.flip(x, (-2,)).transpose(-1, -2)  # noqa: E731
        Pr = torch.stack([turn(P[0]), turn(P[2]), -turn(P[1]), turn(P[3])])
        G, dG, on, b1, b2 = self.sweep(Pr, turn(A), self.dy, self.dx, dt, flux)
        G, dG = (torch.stack([back(x[0]), -back(x[2]), back(x[1]), back(x[3])]) for x in (G, dG))
        on, b1, b2 = back(on), back(b1), back(b2)
        div = lambda f, g: -(f[..., 1:] - f[..., :-1]) / self.dx - (g[..., 1:, :] - g[..., :-1, :]) / self.dy  # noqa: E731
        a, b = a1 * a2, b1 * b2
        return div(F, G), div(dF, dG), div(om * dF, on * dG), a[:, :-1] * a[:, 1:] * b[:-1] * b[1:]

    def alpha0(self, W):
        return self.stage(W, torch.ones_like(W[0]), 1.0, flux=LF)[3]

    def cfl(self, W):
        rho, u, v, p = self._prim(W)
        c = torch.sqrt(self.s.gamma * p / rho)
        return float(self.s.cfl * torch.minimum(self.dx / (u.abs() + c), self.dy / (v.abs() + c)).min())

    def step(self, W, alpha):
        dt = self.cfl(W.detach())
        L, D, Dt, an = self.stage(W, alpha, dt)
        if self.s.time_scheme == SSPRK3:
            W1 = W + dt * L
            W2 = 0.75 * W + 0.25 * W1 + 0.25 * dt * self.stage(W1, alpha, dt)[0]
            L, _, _, an = self.stage(W2, alpha, dt)
            return W / 3 + 2 * W2 / 3 + 2 * dt / 3 * L, an, dt
        Ws = W + 0.5 * dt * L + 0.125 * dt * dt * D
        _, _, Dts, an = self.stage(Ws, alpha, dt)
        return W + dt * L + 0.5 * dt * dt * D + dt * dt / 3 * (Dts - Dt), an, dt

    def run(self, W, steps):
        alpha, t = self.alpha0(W.detach()), 0.0
        for _ in range(steps):
            W, alpha, dt = self.step(W, alpha)
            alpha, t = alpha.detach(), t + dt
        return W, alpha, t


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    put = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    s, d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        with torch.no_grad():
            return [_Scheme(q, dev).run(put(W), case["steps"])[:2] for q, W in zip(s, d)]
    M = _Scheme(s, dev)
    if kind in ("run", "blocks"):
        with torch.no_grad():
            W, a, t = M.run(put(d["W"]), case["steps"])
        return {"W": W, "alpha": a, "t": t, "step": case["steps"]}
    if kind == "stage":
        with torch.no_grad():
            return list(M.stage(put(d["W"]), put(d["alpha"]), _stage_dt(s)))
    W0 = put(d["W"]).requires_grad_(True)
    if kind == "vjp":
        out = M.stage(W0, put(d["alpha"]), _stage_dt(s))[:3]
        torch.autograd.backward(list(out), [put(b) for b in d["bars"]])
        return W0.grad
    W, _, _ = M.run(W0, case["steps"])
    W.backward(put(d["bar"]))
    return {"W": W.detach(), "gradient": W0.grad}
