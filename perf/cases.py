"""The solves whose time counts, through the package's public entry points.

One pass is what a user's program does for one solve: set the initial profile, take the steps,
read the final profile (and, for the bounded grids, hand over the boundary values).  The handle
(``Solver``, ``Batch`` or ``Server``) is made once in ``prepare`` and kept, as such a program
keeps it.  Inputs come from the seed: soliton speeds and places, equation coefficients, relaxation
times.  Equations, time steps and relaxation times are those of ``workloads.py`` and of the tests.

Results are returned in the type that the chosen path computes in: FP64 runs as float64, FP32 runs
(whose phi is a single-precision number, widened by the readout) as float32.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0907_1720_gb300 import lbhpde as L
from paper_0907_1720_gb300 import workloads as W

# dt, tau and spacing of each periodic equation (workloads.py)
EQUATIONS = {
    "kdv": dict(make=W.kdv, dt=1e-5, tau=1.1, b=5, D=5),
    "ks": dict(make=W.ks, dt=1e-4, tau=1.3, b=5, D=5),
    "kawahara": dict(make=W.kawahara, dt=1e-4, tau=2.02, b=7, D=7),
    "gkdv": dict(make=lambda: W.gkdv(1.5), dt=1e-4, tau=1.3, b=5, D=9),
}
DX = 0.1
# bounded grids with stable settings (tests): Example 4.1 on D1Q5, Example 4.5 on D1Q7
BOUNDED = {
    "4.1": dict(make=W.ks, exact=W.ks_shock, dt=1e-3, tau=(1.989, 2.6), scheme=1 | L.NO_AUX_CORRECTION, depth=2, b=5, D=5),
    "4.5": dict(make=W.kawahara, exact=W.kawahara_soliton, dt=1e-4, tau=(2.02, 2.6), scheme=1, depth=1, b=7, D=7),
}


def listed():
    return [
        # the smallest solve anybody runs: one KdV soliton on 400 nodes in double precision, whose
        # time is that of one step after another
        dict(name="kdv_400_fp64", kind="grid", eq="kdv", N=400, fp64=True, steps=2000),
        # one Kuramoto-Sivashinsky solve on 1024 nodes in the single-precision path
        dict(name="ks_1024_fp32", kind="grid", eq="ks", N=1024, fp64=False, steps=4000),
        # one ragged grid that neither fits one thread block nor fills the chip, on D1Q7
        dict(name="kawahara_50021_fp32", kind="grid", eq="kawahara", N=50021, fp64=False, steps=1000),
        # the batched production run: KdV-Burgers members of 256 to 8192 nodes, host to host
        dict(name="ensemble_4096_fp32", kind="ensemble", count=4096, fp64=False, steps=1000),
        # the same family as a reference run in double precision
        dict(name="ensemble_256_fp64", kind="ensemble", count=256, fp64=True, steps=200),
        # the long single grid, in both precisions
        dict(name="kawahara_2e24_fp32", kind="grid", eq="kawahara", N=1 << 24, fp64=False, steps=256),
        dict(name="kawahara_2000003_fp64", kind="grid", eq="kawahara", N=2000003, fp64=True, steps=100),
        # a search for the best relaxation time on the paper's bounded grid (Example 4.1)
        dict(name="tau_sweep_5928_fp32", kind="sweep", example="4.1", count=5928, N=601, fp64=False, steps=500),
        # the same on D1Q7 in double precision (Example 4.5)
        dict(name="tau_sweep_304_fp64", kind="sweep", example="4.5", count=304, N=601, fp64=True, steps=300),
        # one bounded grid longer than a thread block holds, a refinement of Example 4.5
        dict(name="bounded_3001_fp64", kind="sweep", example="4.5", count=1, N=3001, fp64=True, steps=500),
        # a real exponent in the flux: u^1.5 u_x
        dict(name="gkdv_2e22_fp32", kind="grid", eq="gkdv", N=1 << 22, fp64=False, steps=200),
        # a burst of mixed requests to the server: 128 to 65536 nodes each, five equations
        dict(name="serving_48_fp32", kind="serving", count=48, fp64=False, lo=1000, hi=10000),
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(("small", "small", "grid", "grid", "ensemble", "ensemble", "sweep", "bounded", "serving"))
    fp64 = rng.random() < 0.4
    if kind in ("small", "grid"):
        eq = rng.choice(("kdv", "ks", "kawahara", "gkdv"))
        if kind == "small":
            N = _log_int(rng, 64, 6000)
            return dict(kind="grid", eq=eq, N=N, fp64=fp64, steps=rng.randint(200, min(3000, int(2.5e6 / N)) if fp64 else 3000))
        # a grid's cost: at most that of the largest listed one of its precision
        N = _log_int(rng, 6001, 1 << 24)
        most = (2e8 if eq != "gkdv" else 8e7) if fp64 else (4e9 if eq != "gkdv" else 8e8)
        return dict(kind="grid", eq=eq, N=N, fp64=fp64, steps=max(3, min(1500, int(most / N))))
    if kind == "ensemble":
        count = _log_int(rng, 8, 384 if fp64 else 4096)
        return dict(kind="ensemble", count=count, fp64=fp64, steps=rng.randint(50, 200 if fp64 else 1000))
    if kind == "sweep":
        ex = rng.choice(("4.1", "4.5"))
        count = _log_int(rng, 4, 304 if fp64 or ex == "4.5" else 5928)
        return dict(kind="sweep", example=ex, count=count, N=rng.randint(301, 1500 if fp64 or ex == "4.5" else 601), fp64=fp64,
                    steps=rng.randint(50, 150 if fp64 else 300))
    if kind == "bounded":
        return dict(kind="sweep", example=rng.choice(("4.1", "4.5")), count=1, N=_log_int(rng, 2049, 20000), fp64=fp64,
                    steps=rng.randint(100, 500))
    return dict(kind="serving", count=rng.randint(8, 48), fp64=False, lo=1000, hi=rng.randint(2000, 10000))


# ------------------------------------------------------------------------------- inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _sech(z):
    return 1.0 / torch.cosh(z.clamp(-350.0, 350.0))


def _grid_profile(case, seed):
    """[N] initial profile of a periodic grid, on the device."""
    rng = np.random.default_rng([seed, case["N"]])
    N, eq = case["N"], case["eq"]
    x = torch.arange(N, dtype=torch.float64, device=_device()) * DX
    L_ = N * DX
    if eq == "ks":
        k = max(1, round(L_ / 100.0))  # waves of about the length of the 32 pi domain
        z = 2.0 * math.pi * k * x / L_ + float(rng.uniform(0.0, 2.0 * math.pi))
        return float(rng.uniform(0.7, 1.0)) * torch.cos(z) * (1.0 + torch.sin(z))
    # a train of solitary waves, one per 60 length units at most, of random place and size
    period = L_ / max(1, int(L_ // 60.0))
    s = float(rng.uniform(0.0, period))
    z = torch.remainder(x - s, period) - 0.5 * period
    if eq == "kdv":
        c = float(rng.uniform(1.0, 4.0))
        return 0.5 * c * _sech(0.5 * math.sqrt(c) * z) ** 2
    if eq == "gkdv":
        c, n = float(rng.uniform(0.7, 1.0)), 1.5
        return 0.05 + (c * (n + 1.0) * (n + 2.0) / 2.0 * _sech(0.5 * n * math.sqrt(c) * z) ** 2) ** (1.0 / n)
    a = float(rng.uniform(0.5, 1.0))
    return a * 105.0 / 169.0 * _sech(0.5 * math.sqrt(1.0 / 13.0) * z) ** 4


def _grid_problem(case):
    e = EQUATIONS[case["eq"]]
    return W.Problem(e["make"](), case["N"], DX, e["dt"], e["tau"], case["steps"], None)


def _ensemble_problems(case, seed):
    # the sizes belong to the case, the equations and solitons to the seed
    sizes = np.random.default_rng(case["count"]).integers(256, 8193, case["count"])
    rng = np.random.default_rng([seed, case["count"]])
    out = []
    for N in sizes.tolist():
        a, b, d, c = (float(rng.uniform(*r)) for r in ((1.0, 6.0), (0.0, 0.1), (0.5, 1.0), (1.0, 4.0)))
        out.append(W.Problem(W.kdv_burgers(a, b, d), N, W.ENSEMBLE_DX, W.ENSEMBLE_DT, W.ENSEMBLE_TAU, case["steps"], None,
                             meta={"a": a, "d": d, "c": c}))
    return out


def _ensemble_profile(problems):
    """The members' solitons, concatenated, on the device."""
    dev = _device()
    n = torch.tensor([p.N for p in problems], device=dev)

    def each(v):
        return torch.tensor(v, dtype=torch.float64, device=dev).repeat_interleave(n)

    start = (torch.cumsum(n, 0) - n).repeat_interleave(n)
    x = (torch.arange(int(n.sum()), device=dev) - start).double() * W.ENSEMBLE_DX - 0.5 * W.ENSEMBLE_DX * n.repeat_interleave(n).double()
    amp = each([3.0 * p.meta["c"] / p.meta["a"] for p in problems])
    wid = each([0.5 * math.sqrt(p.meta["c"] / p.meta["d"]) for p in problems])
    return amp * _sech(wid * x) ** 2


def _sweep_problems(case, seed):
    """One problem per relaxation time (shared grid and boundary values), and phib [steps, 2W]."""
    e = BOUNDED[case["example"]]
    rng = np.random.default_rng([seed, case["N"]])
    N, n = case["N"], case["steps"]
    xl = -0.5 * (N - 1) * DX + float(rng.uniform(-1.0, 1.0))
    x = W.grid(xl, N, DX)
    taus = np.sort(rng.uniform(e["tau"][0], e["tau"][1], case["count"])) if case["count"] > 1 else [e["tau"][0]]
    ps = [W.Problem(e["make"](), N, DX, e["dt"], float(t), n, e["exact"](x, 0.0), xl=xl, scheme=e["scheme"], boundary="nee",
                    exact_xt=e["exact"], meta={"depth": e["depth"]}) for t in taus]
    return ps, W.boundary_values(ps[0], (e["b"] - 1) // 2, 0, n)


def _requests(case, seed):
    # sizes, equations and step counts belong to the case, the profiles' heights to the seed
    rng = np.random.default_rng([seed, case["count"]])
    ps = [p for _, p in W.serving_requests(case["count"], seed=case["count"], s_lo=case["lo"], s_hi=case["hi"])]
    for p in ps:
        p.phi0 = p.phi0 * float(rng.uniform(0.8, 1.0))
    return ps


def _precision(case):
    return L.FP64 if case["fp64"] else L.FP32_DEV


def prepare(case, seed):
    kind, prec = case["kind"], _precision(case)
    if kind == "grid":
        phi0 = _grid_profile(case, seed)
        return dict(case=case, solver=L.Solver.for_problem(_grid_problem(case), precision=prec), phi0=phi0, out=torch.empty_like(phi0))
    if kind == "ensemble":
        ps = _ensemble_problems(case, seed)
        phi0 = _ensemble_profile(ps).cpu()
        return dict(case=case, batch=L.Batch(ps, precision=prec), phi0=phi0.pin_memory(),
                    out=torch.empty_like(phi0).pin_memory())
    if kind == "sweep":
        ps, phib = _sweep_problems(case, seed)
        phi0 = torch.from_numpy(np.tile(ps[0].phi0, len(ps))).cuda()
        return dict(case=case, batch=L.Batch(ps, precision=prec), phi0=phi0, phib=torch.from_numpy(phib).cuda(),
                    out=torch.empty_like(phi0))
    return dict(case=case, server=L.Server(precision=prec, device_bytes=256 << 20, max_active=256),
                problems=_requests(case, seed))


def run(state):
    case = state["case"]
    n = case.get("steps")
    kind = case["kind"]
    if kind == "serving":  # a burst: everything is submitted, then each result is waited for
        srv = state["server"]
        ids = [srv.submit_problem(p) for p in state["problems"]]
        res = [srv.wait(i) for i in ids]
        return [_typed(case, phi) for _, phi, _ in res] + [np.array([status for status, _, _ in res])]
    if kind == "grid":
        return _typed(case, state["solver"].set_phi(state["phi0"]).step(n).read_phi(state["out"]))
    b = state["batch"].set_phi(state["phi0"])
    if kind == "ensemble":  # host to host, with the conservation record of every member
        d = b.step(n).diagnostics()
        phi = b.read_phi(state["out"])
        return [_typed(case, phi), _typed(case, d["sum_phi"]), _typed(case, d["max_abs_phi"]), d["nonfinite"]]
    return _typed(case, b.step_nee(n, state["phib"]).read_phi(state["out"]))


def _typed(case, x):
    if case["fp64"]:
        return x
    return x.float() if isinstance(x, torch.Tensor) else np.asarray(x, dtype=np.float32)


def _per_node(eqb, D):
    return (eqb - 1) * (2 * (D + 1) + 2)  # multiply-adds of the relaxation, flux difference and its sum


def work(case):
    kind = case["kind"]
    if kind == "grid":
        e = EQUATIONS[case["eq"]]
        return {"bytes": 16.0 * case["N"], "flops": float(case["N"]) * case["steps"] * _per_node(e["b"], e["D"])}
    if kind == "ensemble":
        nodes = float(np.random.default_rng(case["count"]).integers(256, 8193, case["count"]).sum())
        return {"bytes": 16.0 * nodes, "flops": nodes * case["steps"] * _per_node(5, 5)}
    if kind == "sweep":
        e, nodes = BOUNDED[case["example"]], float(case["N"]) * case["count"]
        return {"bytes": 16.0 * nodes + 8.0 * (e["b"] - 1) * case["steps"], "flops": nodes * case["steps"] * _per_node(e["b"], e["D"])}
    # mean of a logarithmically uniform length on [128, 65536] and of uniform steps
    nodes = case["count"] * (65536 - 128) / math.log(65536 / 128)
    return {"bytes": 16.0 * nodes, "flops": nodes * 0.5 * (case["lo"] + case["hi"]) * (0.8 * _per_node(5, 5) + 0.2 * _per_node(7, 7))}


# ------------------------------------------------------------------------- in 64 bits
# The scheme as the paper writes it (collide, stream, zeroth moment), every population stored, in
# plain torch operations on float64.  A polynomial in phi and w = phi^nu is a dict
# {(i, a): coefficient of phi^i w^a}.

def _mul(p, q):
    r = {}
    for (i, a), u in p.items():
        for (k, b), v in q.items():
            r[i + k, a + b] = r.get((i + k, a + b), 0.0) + u * v
    return r


def _add(*terms):
    r = {}
    for s, p in terms:
        for k, u in p.items():
            r[k] = r.get(k, 0.0) + s * u
    return r


def _power(p, k):
    r = {(0, 0): 1.0}
    for _ in range(k):
        r = _mul(r, p)
    return r


def _equilibria(p):
    """(b, [f^eq_0 .. f^eq_{b-1}]) of a problem: Secs. II and III of the paper."""
    eq = p.eq
    m, nu = eq.m, eq.nu
    no_aux, scheme = bool(p.scheme & 0x100), p.scheme & 0xff
    b = eq.lattice or (5 if m <= 4 else 7)
    dt, c, tau = p.dt, p.dx / p.dt, p.tau
    Pi = {k: {} for k in range(1, 7)}
    for k in range(1, m + 1):
        Pi[k] = {(i, 0): float(v) for i, v in enumerate(eq.pi[k - 1]) if v}
        if eq.pi_nu:
            Pi[k].update({(i, 1): float(v) for i, v in enumerate(eq.pi_nu[k - 1]) if v})
    Pi[1] = _add((eq.alpha[0], Pi[1]))
    # tau_k: Taylor coefficients of (e^z - 1) / (1 + tau (e^z - 1)), with alternating sign
    ez = [1.0 / math.factorial(i) for i in range(8)]
    t = [0.0] * 7
    for k in range(1, 7):
        t[k] = ez[k] - tau * sum(ez[i] * t[k - i] for i in range(1, k))
    beta = [0.0] * 7
    for k in range(2, m + 1):
        if eq.alpha[k - 1] and Pi[k]:
            beta[k] = eq.alpha[k - 1] / (dt ** (k - 1) * t[k])
    _, t1, t2, t3, t4, t5, t6 = t
    _, _, b2, b3, b4, b5, _ = beta
    A4 = A5 = A6 = 0.0
    if not no_aux:
        if b2:
            A4 = t2 * (3 * t3 - t2 * t2) * b2 * b2 / t4
        if b == 7 and b2 and b3:
            A5 = (4 * t2 * t4 + 3 * t3 * t3 - 2 * t2 * t2 * t3) * b2 * b3 / t5
        if b == 7 and (b2 or b3):
            A6 = ((5 * t2 * t5 + 3 * t3 * t4 - 2 * t2 * t2 * t4) * b2 * b4 + (4 * t4 - t2 * t3) * t3 * b3 * b3
                  + (t2 * t3 - 6 * t4) * t2 * t2 * b2 ** 3) / t6
    d = {k: {(i - 1, a): (i + a * nu) * v for (i, a), v in Pi[k].items() if i} for k in Pi}
    q = [_power(d[1], k) for k in range(7)]

    def integral(g):
        return {(i + 1, a): v / (i + 1 + a * nu) for (i, a), v in g.items()}

    one = {(0, 0): 1.0}
    aux = {
        2: integral(q[2]),
        3: integral(_add((1, q[3]), (3 * b2, _mul(d[2], q[1])))),
        4: integral(_add((1, q[4]), (6 * b2, _mul(d[2], q[2])), (4 * b3, _mul(d[3], q[1])), (A4, one))),
        5: integral(_add((1, q[5]), (10 * b2, _mul(d[2], q[3])), (10 * b3, _mul(d[3], q[2])), (5 * b4, _mul(d[4], q[1])), (A5, one))),
        6: integral(_add((1, q[6]), (15 * b2, _mul(d[2], q[4])), (20 * b3, _mul(d[3], q[3])), (15 * b4, _mul(d[4], q[2])),
                         (6 * b5, _mul(d[5], q[1])), (A6, one))),
    }
    P = [{(1, 0): 1.0}, _add((1 / c, Pi[1]))] + [_add((c ** -k, aux[k]), (beta[k] * c ** -k, Pi[k])) for k in range(2, b)]
    if scheme == 2:
        P[b - 1] = {}
    # f^eq = M^-1 Pibar with M the Vandermonde matrix of the velocities
    e = np.array([0, 1, -1, 2, -2, 3, -3][:b], dtype=np.float64)
    inv = np.round(np.linalg.inv(np.vander(e, increasing=True).T) * 720) / 720
    return b, [_add(*((inv[j, k], P[k]) for k in range(b))) for j in range(b)]


class _Exact:
    """Several problems of one lattice side by side, concatenated."""

    def __init__(self, problems, phi0):
        self.ps, self.n = problems, [p.N for p in problems]
        dev = _device()
        models = [_equilibria(p) for p in problems]
        self.b, self.W = models[0][0], (models[0][0] - 1) // 2
        self.e = [0, 1, -1, 2, -2, 3, -3][: self.b]
        N = torch.tensor(self.n, device=dev)
        first = torch.cumsum(N, 0) - N
        self.first = first.tolist()
        at = torch.arange(int(N.sum()), device=dev)
        s, n = first.repeat_interleave(N), N.repeat_interleave(N)
        self.source = [None] + [s + torch.remainder(at - s - v, n) for v in self.e[1:]]
        self.nu = problems[0].eq.nu
        keys = sorted({k for _, f in models for g in f for k in g})
        self.top = max(i for i, _ in keys)
        self.rows = max(a for _, a in keys)
        self.member = torch.arange(len(problems), device=dev).repeat_interleave(N)

        def spread(v):
            v = torch.tensor(v, dtype=torch.float64, device=dev)
            return v[0] if len(problems) == 1 else v

        self.coef = [[[spread([f[j].get((i, a), 0.0) for _, f in models]) for i in range(self.top + 1)] for a in range(self.rows + 1)]
                     for j in range(self.b)]
        self.omega = spread([1.0 / p.tau for p in problems])
        if len(problems) > 1:
            self.omega = self.omega[self.member]
            if len(at) * self.b * (self.top + 1) * (self.rows + 1) < 8e9:  # a coefficient per node where that fits
                self.coef = [[[c[self.member] for c in r] for r in rows] for rows in self.coef]
                self.member = None
        else:
            self.member = None
        self.f = [g.clone() for g in self.feq(phi0.to(dev))]

    def _c(self, c, member):
        return c if member is None else c[member]

    def feq(self, phi, at=None):
        """f^eq_j(phi); at: the concatenated places of the nodes that phi stands for."""
        m = self.member if at is None or self.member is None else self.member[at]
        w = torch.where(phi > 0, phi.clamp(min=1e-300) ** self.nu, torch.zeros_like(phi)) if self.rows else None
        out = []
        for rows in self.coef:
            acc = None
            for r in reversed(rows):
                h = torch.zeros_like(phi)
                for c in reversed(r):
                    c = self._c(c, m)
                    c = c[at] if at is not None and m is None and c.ndim else c
                    h = h * phi + c
                acc = h if acc is None else acc * w + h
            out.append(acc)
        return out

    def step(self, live=None):
        phi = sum(self.f)
        new = []
        for j, (f, g) in enumerate(zip(self.f, self.feq(phi))):
            s = f - (f - g) * self.omega
            s = s if j == 0 else s[self.source[j]]
            new.append(s if live is None else torch.where(live, s, f))
        self.f = new

    def bound(self, phib, depth):
        """The outer nodes from the prescribed values phib [2W] (shared by all members)."""
        dev = phib.device
        first, N = torch.tensor(self.first, device=dev), torch.tensor(self.n, device=dev)
        for side in (0, 1):
            xf = first + (self.W - 1 + depth) if side == 0 else first + N - self.W - depth
            inner = self.feq(sum(f[xf] for f in self.f), xf)
            for l in range(self.W):
                x = first + l if side == 0 else first + N - self.W + l
                outer = self.feq(phib[side * self.W + l].expand(len(self.n)).contiguous(), x)
                for j in range(self.b):
                    self.f[j][x] = outer[j] + self.f[j][xf] - inner[j]

    def phi(self):
        return sum(self.f)


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid":
        E = _Exact([_grid_problem(case)], _grid_profile(case, seed))
        for _ in range(case["steps"]):
            E.step()
        return E.phi()
    if kind == "ensemble":
        ps = _ensemble_problems(case, seed)
        E = _Exact(ps, _ensemble_profile(ps))
        for _ in range(case["steps"]):
            E.step()
        phi = E.phi()
        parts = phi.split(E.n)
        return [phi, torch.stack([p.sum() for p in parts]), torch.stack([p.abs().max() for p in parts]), None]
    if kind == "sweep":
        ps, phib = _sweep_problems(case, seed)
        E = _Exact(ps, torch.from_numpy(np.tile(ps[0].phi0, len(ps))))
        phib = torch.from_numpy(phib).to(_device())
        for row in phib:
            E.step()
            E.bound(row, ps[0].meta["depth"])
        return E.phi()
    ps = _requests(case, seed)
    got = [None] * len(ps)
    for lattice in (5, 7):
        which = [i for i, p in enumerate(ps) if (7 if p.eq.m > 4 else 5) == lattice]
        if not which:
            continue
        sub = [ps[i] for i in which]
        E = _Exact(sub, torch.from_numpy(np.concatenate([p.phi0 for p in sub])))
        steps = torch.tensor([p.nsteps for p in sub], device=_device())
        left = steps.repeat_interleave(torch.tensor(E.n, device=_device()))
        shortest, longest = min(p.nsteps for p in sub), max(p.nsteps for p in sub)
        for s in range(longest):
            E.step(None if s < shortest else left > s)
        for i, phi in zip(which, E.phi().split(E.n)):
            got[i] = phi
    return got + [None]
