"""Performance cases of the momentum-loop library: what its users call, over the sizes they use.

Every case goes through the public binding (Context.rhs, ft_states, flow, serving, and the
differentiable rhs of autograd).  Table profiles are smooth bumps on the logarithmic momentum grid,
seeded; grids and quadrature orders are those of the benchmark, the tests and the serving mix, with
ragged ones between them.

`exact` is the same discrete sum in plain FP64 tensor arithmetic.  Adaptive flows have none: their
endpoints depend on the step sequence.
"""
import math
import time
from types import SimpleNamespace

import numpy as np
import torch

import paper_2412_13043_gb300 as ffrg
from paper_2412_13043_gb300 import autograd

D3, D4, FT, D4F, FT4 = (ffrg.MODEL_D3, ffrg.MODEL_D4_VERTEX, ffrg.MODEL_FINITE_T, ffrg.MODEL_D4_FULL,
                        ffrg.MODEL_FINITE_T_4D)
PRECISION = {"fp64": ffrg.FP64, "mixed": ffrg.MIXED}
X_MIN, X_MAX, QMAX = 1e-3, 10.0, 4.0   # table and external grid, radial domain in units of k
LAMBDA = 10.0                          # UV scale of the flows


# --------------------------------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------------------------------
def listed():
    return [
        # one d=3 two-point right-hand side of a small truncation in the default precision: the
        # smallest call, as a user's own stepper or a test makes it
        dict(name="d3 rhs small", kind="d3", precision="fp64", n_pts=64, n_ext=16, n_rad=32, n_ang=16, flat=False,
             m2=0.5, k=1.0),
        # the d=3 two-point flow k = 10 -> 0.01 at the benchmark's size and tolerance (about 200
        # right-hand sides inside one call)
        dict(name="d3 flow", kind="flow_d3", precision="fp64", feedback=False, n_pts=64, n_ext=64, n_rad=64,
             n_ang=32, m2=0.5, k_end=0.01, rtol=1e-10),
        # the d=4 vertex expansion, mixed precision: the benchmark's headline workload
        dict(name="d4 rhs mixed", kind="d4", precision="mixed", n_pts=128, n_ext_ang=8, n_rad=128, n_ang1=64,
             n_ang2=16, flat=False, M2=1.0, k=1.0),
        # the same truncation in the library's default precision (reference runs, stiff flows)
        dict(name="d4 rhs fp64", kind="d4", precision="fp64", n_pts=128, n_ext_ang=8, n_rad=128, n_ang1=64,
             n_ang2=16, flat=False, M2=1.0, k=1.0),
        # the full three-point vertex on the 96 x 8 x 7 grid, mixed
        dict(name="d4 full rhs mixed", kind="d4full", precision="mixed", n_pts=96, n_va=8, n_vb=7, n_ext_ang=8,
             n_rad=128, n_ang1=64, n_ang2=16, flat=False, M2=1.0, k=1.0),
        # finite temperature, bosonic, mixed, at the benchmark's N = 16
        dict(name="finite T rhs mixed", kind="ft", precision="mixed", N=16, T=0.002, n_pts=64, n_ext_p=64,
             n_ext_m=9, n_rad=96, n_ang=48, fermi=False, flat=False, m2=0.5, k=1.0),
        # finite temperature, fermionic, default precision, ragged sizes as a parameter scan has them
        dict(name="finite T rhs fp64 ragged", kind="ft", precision="fp64", N=33, T=0.01, n_pts=97, n_ext_p=51,
             n_ext_m=7, n_rad=77, n_ang=39, fermi=True, flat=False, m2=0.3, k=0.7),
        # finite temperature with the 4D regulator: 25 loop frequencies in the domain at k = 1
        dict(name="finite T 4D rhs fp64", kind="ft4", precision="fp64", N=16, T=0.05, n_pts=64, n_ext_p=64,
             n_ext_m=9, n_rad=96, n_ang=48, n_x0=64, fermi=False, flat=False, m2=0.5, k=1.0),
        # 1024 loop-side states against one angle-integrated kernel (tensor cores)
        dict(name="finite T states", kind="states", precision="fp64", N=16, T=0.002, n_pts=64, n_ext_p=64,
             n_ext_m=9, n_rad=96, n_ang=48, fermi=False, flat=False, m2=0.5, k=1.0, n_states=1024),
        # value and gradient with respect to the tables, forward and backward through autograd
        dict(name="d4 value and gradient", kind="d4grad", n_pts=96, n_ext_ang=4, n_rad=96, n_ang1=48, n_ang2=16,
             flat=False, M2=1.0, k=1.0),
        # the coupled d=4 flow whose state is its tables, at the stepper comparison's size
        dict(name="d4 feedback flow", kind="flow_d4", precision="fp64", n_pts=32, n_ext_ang=4, n_rad=32, n_ang1=16,
             n_ang2=8, M2=1.0, k_end=0.01, rtol=1e-6),
        # a batch of flow requests of the serving mix, submitted at once to a running server
        dict(name="serving batch", kind="serve", n_requests=48, max_slots=64, t_max=1.0, rtol=1e-10),
    ]


def draw(rng):
    """One more case of the same ranges; sizes log-uniform, often odd."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    kind = rng.choice(["d3", "d4", "d4full", "ft", "ft4", "states", "d4grad", "flow_d3", "flow_d4", "serve"])
    c = dict(kind=kind)
    if kind in ("d3", "d4", "d4full", "ft", "ft4", "states", "flow_d3"):
        c["precision"] = rng.choice(["fp64", "mixed"])
    if kind in ("d3", "d4", "d4full", "ft", "ft4", "states", "d4grad"):
        # the flat regulator is the closed-form check of the default precision
        c["flat"] = c.get("precision", "fp64") == "fp64" and rng.random() < 0.25
        c["k"] = log(0.02, 10.0)
    if kind == "d3":
        c.update(n_pts=size(16, 256), n_ext=size(16, 256), n_rad=size(16, 128), n_ang=size(8, 64),
                 m2=rng.uniform(-0.2, 1.0))
    elif kind in ("d4", "d4grad"):
        c.update(n_pts=size(16, 128 if kind == "d4" else 96), n_ext_ang=size(2, 8 if kind == "d4" else 4),
                 n_rad=size(16, 128 if kind == "d4" else 96), n_ang1=size(8, 64 if kind == "d4" else 48),
                 n_ang2=size(4, 16), M2=rng.uniform(0.0, 1.0))
    elif kind == "d4full":
        c.update(n_pts=size(16, 96), n_va=rng.randint(2, 8), n_vb=rng.randint(2, 7), n_ext_ang=size(2, 8),
                 n_rad=size(16, 128), n_ang1=size(8, 64), n_ang2=size(4, 16), M2=rng.uniform(0.0, 1.0))
        if c["precision"] == "fp64":   # no larger than a quarter of the listed size
            c.update(n_rad=size(16, 64), n_ang1=size(8, 32))
    elif kind in ("ft", "states"):
        c.update(N=rng.randint(1, 64 if kind == "ft" else 32), T=log(0.002, 0.5), n_pts=size(16, 160),
                 n_ext_p=size(4, 64), n_ext_m=rng.randint(1, 9), n_rad=size(16, 128), n_ang=size(8, 64),
                 fermi=rng.random() < 0.4, m2=rng.uniform(-0.2, 1.0))
        if kind == "states":
            c["n_states"] = size(32, 1024)
    elif kind == "ft4":
        c.update(N=rng.randint(2, 24), T=min(log(0.01, 0.5), 0.2 * c["k"]), n_pts=size(16, 160), n_ext_p=size(4, 64),
                 n_ext_m=rng.randint(1, 9), n_rad=size(16, 96), n_ang=size(8, 48), n_x0=size(8, 64),
                 fermi=rng.random() < 0.4, m2=rng.uniform(-0.2, 1.0))
    elif kind == "flow_d3":
        c.update(feedback=False, n_pts=size(32, 128), n_ext=size(16, 96), n_rad=size(24, 96), n_ang=size(12, 48),
                 m2=rng.uniform(0.1, 1.0), k_end=log(0.01, 1.0), rtol=log(1e-10, 1e-7))
    elif kind == "flow_d4":
        c.update(precision="fp64", n_pts=size(16, 32), n_ext_ang=size(2, 4), n_rad=size(16, 32), n_ang1=size(8, 16),
                 n_ang2=size(4, 8), M2=rng.uniform(0.5, 1.0), k_end=log(0.01, 0.5), rtol=1e-6)
    else:
        c.update(n_requests=rng.randint(8, 48), max_slots=rng.choice([16, 32, 64]), t_max=rng.choice([0.005, 1.0]),
                 rtol=log(1e-10, 1e-8))
    if c.get("fermi") and kind == "ft4":
        c["n_ext_m"] = 1   # one external fermion frequency
    return c


# --------------------------------------------------------------------------------------------------
# inputs: the problem and its tables from a case and a seed
# --------------------------------------------------------------------------------------------------
def _grid(n):
    return X_MIN * (X_MAX / X_MIN) ** (np.arange(n) / (n - 1)) if n > 1 else np.array([X_MIN])


def _bump(x2, amp, width):
    return 1.0 + amp * np.exp(-x2 / width)


def _profiles(rng):
    u = rng.uniform
    return SimpleNamespace(a=u(0.0, 0.2), b=u(0.5, 2.0), g3=u(0.5, 1.5), c3=u(-0.3, 0.3), b3=u(0.5, 2.0),
                           g4=u(0.5, 1.5), c4=u(-0.3, 0.3), b4=u(0.5, 2.0), ea=u(-0.2, 0.2), eb=u(-0.2, 0.2),
                           eab=u(-0.1, 0.1))


def _problem(c):
    """The problem of a case, with the attributes that the binding reads."""
    kind = c["kind"]
    model = {"d3": D3, "flow_d3": D3, "d4": D4, "d4grad": D4, "flow_d4": D4, "d4full": D4F, "ft": FT, "states": FT,
             "ft4": FT4}[kind]
    p = SimpleNamespace(model=model, regulator=ffrg.REG_LITIM if c.get("flat") else ffrg.REG_EXP, n_rad=c["n_rad"],
                        n_ang1=c.get("n_ang1", c.get("n_ang")), n_ang2=c.get("n_ang2", 1),
                        n_ext_p=c.get("n_ext_p", c.get("n_ext", c["n_pts"])), n_ext_ang=c.get("n_ext_ang", 1),
                        n_matsubara=c.get("N", 0), include_p0=0, statistics=1 if c.get("fermi") else 0,
                        m2_over_k2=c.get("m2", 0.5), m2_shift=c.get("M2", 0.0), lam=1.0, T=c.get("T", 0.0),
                        p_min=X_MIN, p_max=X_MAX, qmax_over_k=QMAX, prefactor=1.0, n_va=c.get("n_va", 1),
                        n_vb=c.get("n_vb", 1), n_x0=c.get("n_x0", 0), n_tables=1, n_stack=1, n_pts=c["n_pts"],
                        x_min=X_MIN, x_max=X_MAX)
    if model in (FT, FT4):
        p.n_ext_ang, p.n_tables = c["n_ext_m"], 2
        p.n_stack = c["N"] + c["n_ext_m"] if model == FT else 1
    elif model in (D4, D4F):
        p.n_tables, p.n_stack = 3, p.n_va * p.n_vb
    return p


def _tables(p, rng):
    f = _profiles(rng)
    x2 = _grid(p.n_pts) ** 2
    if p.model == D3:
        return _bump(x2, f.a, f.b).reshape(1, 1, -1)
    if p.model == FT:
        j = np.arange(p.n_stack)
        om = math.pi * p.T * (2 * j + 1) if p.statistics else 2 * math.pi * p.T * j
        x2 = x2[None, :] + om[:, None] ** 2
        return np.stack([_bump(x2, f.a, f.b), f.g3 * _bump(x2, f.c3, f.b3)])
    if p.model == FT4:
        return np.stack([_bump(x2, f.a, f.b), f.g3 * _bump(x2, f.c3, f.b3)]).reshape(2, 1, -1)
    if p.model == D4:
        return np.stack([_bump(x2, f.a, f.b), f.g3 * _bump(x2, f.c3, f.b3),
                         f.g4 * _bump(x2, f.c4, f.b4)]).reshape(3, 1, -1)
    t = np.zeros((3, p.n_stack, p.n_pts))
    t[0, 0], t[2, 0] = _bump(x2, f.a, f.b), f.g4 * _bump(x2, f.c4, f.b4)
    av, bv = np.linspace(-1, 1, p.n_va), np.linspace(-1, 1, p.n_vb)
    shape = 1 + f.ea * av[:, None] + f.eb * bv[None, :] + f.eab * av[:, None] * bv[None, :]
    t[1] = shape.reshape(-1, 1) * (f.g3 * _bump(x2, f.c3, f.b3))[None, :]
    return t


def _flow_start(p, tables, feedback):
    """Initial state of a flow: the tables (d=4 feedback), or Z(p) p^2 + m^2 at the external points."""
    if feedback:
        return tables.reshape(-1).copy()
    ps = _grid(p.n_ext_p)
    m2 = p.m2_over_k2 * LAMBDA ** 2
    if p.model == D3:
        return np.interp(np.log(ps), np.log(_grid(p.n_pts)), tables[0, 0]) * ps ** 2 + m2
    om = 2 * math.pi * p.T * np.arange(p.n_ext_ang)
    return (ps[:, None] ** 2 + om[None, :] ** 2 + m2).reshape(-1)


def _requests(c, rng):
    """Flow requests of the serving mix: temperatures in [0, t_max], below 0.01 the d=3 family.  The grids
    are the case's, the masses and profiles the seed's."""
    out, mix = [], np.random.RandomState(c["n_requests"])
    for _ in range(c["n_requests"]):
        T = mix.uniform(0.0, c["t_max"])
        n_ext, n_rad, n_ang, n_pts = (int(mix.randint(a, b + 1)) for a, b in ((32, 256), (32, 128), (16, 64), (64, 256)))
        if T < 0.01:
            p = _problem(dict(kind="d3", n_pts=n_pts, n_ext=n_ext, n_rad=n_rad, n_ang=n_ang, m2=rng.uniform(-0.2, 1.0)))
        else:
            N = min(64, math.ceil(LAMBDA / (2 * math.pi * T)))
            p = _problem(dict(kind="ft", N=N, T=T, n_pts=n_pts, n_ext_p=max(1, n_ext // 9), n_ext_m=9, n_rad=n_rad,
                              n_ang=n_ang, m2=rng.uniform(-0.2, 1.0)))
        t = _tables(p, rng)
        out.append((p, t, _flow_start(p, t, False)))
    return out


def _inputs(c, seed):
    """(problem, tables, generator for the case's other inputs)."""
    rng = np.random.RandomState(seed & 0x7FFFFFFF)
    p = _problem(c)
    return p, _tables(p, rng), rng


def _nfreq(p):
    return 2 * p.n_matsubara + 1 + (1 if p.statistics else 0)


def _states(c, p, rng):
    """Loop-side states: decaying profiles over loop frequencies and radial nodes with noise on them."""
    g = torch.Generator().manual_seed(int(rng.randint(1 << 30)))
    n = torch.arange(_nfreq(p), dtype=torch.float64) - p.n_matsubara
    r = (torch.arange(p.n_rad, dtype=torch.float64) + 0.5) / p.n_rad
    shape = torch.exp(-3 * r[None, :] ** 2) / (1 + 0.05 * n[:, None] ** 2)
    return shape[None] * (0.5 + torch.rand(c["n_states"], _nfreq(p), p.n_rad, dtype=torch.float64, generator=g))


def prepare(case, seed):
    c = dict(case)
    ctx = ffrg.Context(torch.cuda.current_device())
    s = SimpleNamespace(case=c, kind=c["kind"], ctx=ctx)
    if s.kind == "serve":
        s.requests = _requests(c, np.random.RandomState(seed & 0x7FFFFFFF))
        ctx.serve_start(max_slots=c["max_slots"])
        return s
    s.problem, tables, rng = _inputs(c, seed)
    s.precision = PRECISION[c.get("precision", "fp64")]
    if s.kind == "d4grad":
        s.table_values = torch.tensor(tables, device="cuda", requires_grad=True)
        s.grad_out = torch.tensor(rng.uniform(-1.0, 1.0, _n_ext(s.problem)), device="cuda")
        return s
    s.tables = ctx.tables(s.problem, tables)
    if s.kind.startswith("flow"):
        s.y0 = torch.tensor(_flow_start(s.problem, tables, s.kind == "flow_d4"), device="cuda")
    if s.kind == "states":
        s.F = _states(c, s.problem, rng).cuda()
    return s


def run(state):
    s, c = state, state.case
    if s.kind == "serve":
        t1 = math.log(LAMBDA / 0.01)
        left = [(i, s.ctx.serve_submit(p, t, y0, LAMBDA, t1, rtol=c["rtol"], atol=1e-13), len(y0))
                for i, (p, t, y0) in enumerate(s.requests)]
        done = {}
        while left:
            still = []
            for i, ticket, n in left:
                code, y, _, _ = s.ctx.serve_poll(ticket, n)
                if code == ffrg.EPENDING:
                    still.append((i, ticket, n))
                elif code != ffrg.OK:
                    raise RuntimeError(ffrg.strerror(code))
                else:
                    done[i] = y
            left = still
            if left:
                time.sleep(2e-4)
        return np.concatenate([done[i] for i in range(len(s.requests))])
    if s.kind == "d4grad":
        out = autograd.rhs(s.table_values, s.ctx, s.problem, c["k"])
        (grad,) = torch.autograd.grad(out, s.table_values, s.grad_out)
        return {"out": out, "grad": grad}
    if s.kind == "states":
        return s.ctx.ft_states(s.problem, s.tables, c["k"], s.F, precision=s.precision)
    if s.kind.startswith("flow"):
        y = s.y0.clone()
        s.ctx.flow(s.problem, s.tables, y, LAMBDA, math.log(LAMBDA / c["k_end"]), feedback=int(s.kind == "flow_d4"),
                   precision=s.precision, rtol=c["rtol"], atol=1e-3 * c["rtol"])
        return y
    return s.ctx.rhs(s.problem, s.tables, c["k"], precision=s.precision)


# --------------------------------------------------------------------------------------------------
# work: table values in, outputs out, and the integrand's arithmetic (a logarithm, exponential,
# root or division counts as one operation)
# --------------------------------------------------------------------------------------------------
def _n_ext(p):
    if p.model == D3:
        return p.n_ext_p
    return p.n_ext_p * p.n_ext_ang if p.model in (FT, FT4) else 2 * p.n_ext_p + 1 + p.n_ext_p * p.n_ext_ang


def _rhs_flops(p, k=1.0):
    """One right-hand side: argument 2, lookup 6, regulator and propagator 7, sum 2 per factor of a term."""
    rows = p.n_rad * p.n_ang1
    if p.model == D3:
        return 17.0 * p.n_ext_p * rows
    if p.model == FT:   # angular sums once per (frequency row, momentum), then the sum over frequencies
        return 23.0 * (p.n_matsubara + p.n_ext_ang) * p.n_ext_p * rows + 2.0 * _n_ext(p) * _nfreq(p) * p.n_rad
    if p.model == FT4:
        return 23.0 * _n_ext(p) * _ft4_frequencies(p, k)[0].size * rows
    lookup = 6.0 if p.model == D4 else 30.0   # the full vertex: shape variables and a trilinear lookup
    three = p.n_ext_p * p.n_ext_ang * rows * (13.0 + lookup + p.n_ang2 * (19.0 + 2.0 * lookup))
    return three + (2 * p.n_ext_p + 1) * rows * (26.0 + lookup)


def work(case):
    c = dict(case)
    if c["kind"] == "serve":   # about 35 accepted steps of six right-hand sides a flow
        reqs = _requests(c, np.random.RandomState(1))
        return {"bytes": sum(8.0 * (t.size + 2 * y.size) for _, t, y in reqs),
                "flops": sum(35 * 6 * _rhs_flops(p) for p, _, _ in reqs)}
    p = _problem(c)
    tables, ne = 8.0 * p.n_tables * p.n_stack * p.n_pts, 8.0 * _n_ext(p)
    flops = _rhs_flops(p, c.get("k", 1.0))
    if c["kind"] == "states":
        kdim, n = _nfreq(p) * p.n_rad, c["n_states"]
        k_build = flops - 2.0 * _n_ext(p) * kdim
        return {"bytes": tables + 8.0 * n * kdim + n * ne, "flops": k_build + 2.0 * n * _n_ext(p) * kdim}
    if c["kind"] == "d4grad":   # the backward pass about twice the value's work
        return {"bytes": 2 * tables + 2 * ne, "flops": 3 * flops}
    if c["kind"].startswith("flow"):
        state = tables if c["kind"] == "flow_d4" else ne
        return {"bytes": tables + 2 * state, "flops": (205 if c["kind"] == "flow_d3" else 115) * flops}
    return {"bytes": tables + ne, "flops": flops}


# --------------------------------------------------------------------------------------------------
# exact: the same discrete sums in plain FP64 tensor arithmetic
# --------------------------------------------------------------------------------------------------
def _gl(n, a, b):
    """Gauss-Legendre rule: numpy's nodes after one Newton step in extended precision."""
    x = np.polynomial.legendre.leggauss(n)[0].astype(np.longdouble)
    p0, p1 = np.ones_like(x), x
    for j in range(2, n + 1):
        p0, p1 = p1, ((2 * j - 1) * x * p1 - (j - 1) * p0) / j
    if n > 1:
        d = n * (p0 - x * p1) / (1 - x * x)
        x = x - p1 / d
        p0, p1 = np.ones_like(x), x
        for j in range(2, n + 1):
            p0, p1 = p1, ((2 * j - 1) * x * p1 - (j - 1) * p0) / j
        d = n * (p0 - x * p1) / (1 - x * x)
    else:
        d = np.ones_like(x)
    w = 2 / ((1 - x * x) * d * d)
    half = np.longdouble(b - a) / 2
    return ((np.longdouble(a) + b) / 2 + half * x).astype(np.float64), (half * w).astype(np.float64)


def _gc2(n):
    th = np.arange(1, n + 1) * math.pi / (n + 1)
    return np.cos(th), math.pi / (n + 1) * np.sin(th) ** 2


def _ft4_frequencies(p, k):
    """Loop frequencies and weights of the k-scaled domain: the Matsubara sum up to the cap, else quadrature."""
    L, T = QMAX * k, p.T
    if p.statistics:
        x = L / (math.pi * T)
        nk = -1 if x < 1 else math.floor((x - 1) / 2)
        n = np.arange(-nk - 1, nk + 1)
        w = (2 * n + 1) * math.pi * T
    else:
        nk = math.floor(L / (2 * math.pi * T))
        w = 2 * math.pi * T * np.arange(-nk, nk + 1)
    if w.size <= _nfreq(p):
        return w, np.full(w.size, T)
    x, wx = _gl(p.n_x0, -L, L)
    return x, wx / (2 * math.pi)


class _Exact:
    """The sums of one problem at scale k; tables: a FP64 tensor [n_tables, n_stack, n_pts]."""

    def __init__(self, p, tables, k, dev):
        self.p, self.t, self.k, self.k2, self.dev = p, tables, k, k * k, dev
        self.m2 = p.m2_over_k2 * k * k + p.m2_shift
        self.us = 0.5 * (p.n_pts - 1) / math.log(p.x_max / p.x_min)
        self.uo = -(p.n_pts - 1) * math.log(p.x_min) / math.log(p.x_max / p.x_min)
        self.q, self.wq = (self.f(v) for v in _gl(p.n_rad, 0.0, QMAX * k))
        self.c, self.v = (self.f(v) for v in (_gc2(p.n_ang1) if p.model in (D4, D4F) else _gl(p.n_ang1, -1, 1)))
        self.ps = self.f(_grid(p.n_ext_p))

    def f(self, a):
        return torch.as_tensor(np.asarray(a), dtype=torch.float64, device=self.dev)

    def pos(self, s2):
        u = (self.us * torch.log(s2.clamp_min(1e-300)) + self.uo).clamp(0.0, self.p.n_pts - 1.0)
        i = u.long().clamp_max(self.p.n_pts - 2)
        return i, u - i

    def look(self, row, s2):
        i, w = self.pos(s2)
        a = row.take(i)
        return a + w * (row.take(i + 1) - a)

    def reg(self, x):
        """r(x) = R/(Z k^2) and its scale derivative."""
        if self.p.regulator == ffrg.REG_LITIM:
            on = (x < 1).double()
            return on * (1 - x), 2 * on
        em = torch.expm1(-x)
        e = torch.exp(-x)
        return -x * e / em, 2 * x * x * e / (em * em)

    def prop(self, Z, s2, om2=0.0):
        return 1.0 / (Z * (om2 + s2 + self.k2 * self.reg(s2 / self.k2)[0]) + self.m2)

    def d3(self):
        p, q2 = self.p, self.q ** 2
        Z = self.look(self.t[0, 0], q2)
        F = self.wq * q2 * Z * self.k2 * self.reg(q2 / self.k2)[1] * self.prop(Z, q2) ** 2
        s2 = (q2[None, :, None] + self.ps[:, None, None] ** 2
              + 2 * self.q[None, :, None] * self.ps[:, None, None] * self.c[None, None, :])
        G = self.prop(self.look(self.t[0, 0], s2), s2)
        return p.lam ** 2 / (4 * math.pi ** 2) * ((G * self.v).sum(2) * F).sum(1)

    def ft_kernel(self, j):
        """K[j][p][r]: the angular sum of lambda G at stack row j."""
        p, row = self.p, min(j, self.p.n_stack - 1)
        om = math.pi * p.T * (2 * j + (1 if p.statistics else 0))
        s2 = (self.q[None, :, None] ** 2 + self.ps[:, None, None] ** 2
              + 2 * self.q[None, :, None] * self.ps[:, None, None] * self.c)
        Z, L = self.look(self.t[0, row], s2), self.look(self.t[1, row], s2)
        return (self.v * L * self.prop(Z, s2, om * om)).sum(2)

    def ft_index(self, n):
        return (n if n >= 0 else -n - 1) if self.p.statistics else abs(n)

    def ft_factor(self, n):
        p, j = self.p, self.ft_index(n)
        row, q2 = min(j, p.n_stack - 1), self.q ** 2
        om = math.pi * p.T * (2 * j + (1 if p.statistics else 0))
        Z, L = self.look(self.t[0, row], q2), self.look(self.t[1, row], q2)
        return Z * self.k2 * self.reg(q2 / self.k2)[1] * self.prop(Z, q2, om * om) ** 2 * L

    def ft(self, F=None):
        """F: states [S, nfreq, n_rad], or the model's own loop factor (one state)."""
        p = self.p
        n0 = -p.n_matsubara - (1 if p.statistics else 0)
        ns = range(n0, n0 + _nfreq(p))
        K = [self.ft_kernel(j) for j in range(p.n_matsubara + p.n_ext_ang)]
        own = F is None
        if own:
            F = torch.stack([self.ft_factor(n) for n in ns])[None]
        B = (F * (self.wq * self.q ** 2)).reshape(F.shape[0], -1)
        out = torch.empty(F.shape[0], p.n_ext_p, p.n_ext_ang, dtype=torch.float64, device=self.dev)
        for m in range(p.n_ext_ang):
            A = torch.stack([K[self.ft_index(n + m)] for n in ns], 1).reshape(p.n_ext_p, -1)
            out[:, :, m] = B @ A.T
        out = p.lam ** 2 * p.T / (4 * math.pi ** 2) * out.reshape(F.shape[0], -1)
        return out[0] if own else out

    def ft4(self):
        p = self.p
        w, ww = (self.f(v) for v in _ft4_frequencies(p, self.k))
        Q2 = w[:, None] ** 2 + self.q[None, :] ** 2
        Z, L = self.look(self.t[0, 0], Q2), self.look(self.t[1, 0], Q2)
        F = (ww[:, None] * self.wq * self.q ** 2 * Z * self.k2 * self.reg(Q2 / self.k2)[1] * self.prop(Z, Q2) ** 2 * L)
        p0 = ([math.pi * p.T * math.exp(-self.k / (math.pi * p.T))] if p.statistics
              else [2 * math.pi * p.T * m for m in range(p.n_ext_ang)])
        out = torch.empty(p.n_ext_p, p.n_ext_ang, dtype=torch.float64, device=self.dev)
        for i in range(p.n_ext_p):
            for m in range(p.n_ext_ang):
                s2 = ((w + p0[m])[:, None, None] ** 2
                      + (self.q[:, None] ** 2 + self.ps[i] ** 2 + 2 * self.q[:, None] * self.ps[i] * self.c)[None])
                Z, L = self.look(self.t[0, 0], s2), self.look(self.t[1, 0], s2)
                out[i, m] = (F * (self.v * L * self.prop(Z, s2)).sum(2)).sum()
        return p.lam ** 2 / (4 * math.pi ** 2) * out.reshape(-1)

    def lam3(self, s1, s2, s3):
        """Three-point vertex at squared leg momenta s1, s2, s3."""
        p, S = self.p, (s1 + s2 + s3) / 3
        if p.model == D4:
            return self.look(self.t[1, 0], S)

        def cell(v, n):
            u = 0.5 * (torch.nan_to_num(v, nan=-1.0).clamp(-1, 1) + 1) * (n - 1)
            i = u.long().clamp_max(n - 2)
            return i, u - i

        i, w = self.pos(S)
        ia, wa = cell((s3 - s1 - s2) / (2 * torch.sqrt(s1 * s2)), p.n_va)
        ib, wb = cell((s1 - s2) / (s1 + s2), p.n_vb)
        t = self.t[1].reshape(-1)

        def at(da, db):
            o = ((ia + da) * p.n_vb + ib + db) * p.n_pts + i
            a = t.take(o)
            return a + w * (t.take(o + 1) - a)

        return (1 - wa) * ((1 - wb) * at(0, 0) + wb * at(0, 1)) + wa * ((1 - wb) * at(1, 0) + wb * at(1, 1))

    def d4(self, grad_out=None):
        """Outputs; with grad_out also the gradient left on self.t (a leaf), point by point."""
        p, q2 = self.p, self.q ** 2
        x2, w2 = (self.f(v) for v in _gl(p.n_ang2, -1, 1))
        xp, _ = _gl(p.n_ext_ang, -1, 1)
        sw2, n = float(w2.sum()), p.n_ext_p
        s1 = torch.sqrt(1 - self.c ** 2)
        norm = 1.0 / (8 * math.pi ** 3)

        def factor():
            Z = self.look(self.t[0, 0], q2)
            F = self.wq * q2 * self.q * Z * self.k2 * self.reg(q2 / self.k2)[1] * self.prop(Z, q2) ** 2
            return F[:, None] * self.v[None, :]

        def point(e):
            three = n < e < n + 1 + n * p.n_ext_ang
            ip = (e - n - 1) // p.n_ext_ang if three else (e if e <= n else e - n - 1 - n * p.n_ext_ang)
            pe = 0.0 if e == n else float(self.ps[ip])
            cp = float(xp[(e - n - 1) % p.n_ext_ang]) if three else 1.0
            p2, Q2 = torch.tensor(pe * pe, dtype=torch.float64, device=self.dev), q2[:, None]
            A2 = (Q2 + p2 + 2 * self.q[:, None] * pe * self.c).clamp_min(0.0)
            GA = self.prop(self.look(self.t[0, 0], A2), A2)
            if e <= n:
                l4 = self.look(self.t[2, 0], (Q2 + p2) * 0.5)
                v = sw2 * (-0.5 * l4 + self.lam3(Q2, A2, p2) ** 2 * GA)
                return norm * (factor() * v).sum()
            if not three:
                l4 = self.look(self.t[2, 0], (Q2 + A2 + 2 * p2) * 0.25)
                return 1.5 * norm * (factor() * sw2 * GA * l4 * l4).sum()
            C2, sp = 2 * p2 * (1 + cp), math.sqrt(1 - cp * cp)
            cos = cp * self.c[:, None] + sp * s1[:, None] * x2[None, :]
            B2 = (q2[:, None, None] + p2 - 2 * self.q[:, None, None] * pe * cos[None]).clamp_min(0.0)
            GB = self.prop(self.look(self.t[0, 0], B2), B2)
            rs = (w2 * GB * self.lam3(Q2[..., None], B2, p2) * self.lam3(A2[..., None], B2, C2)).sum(2)
            return 3 * norm * (factor() * GA * self.lam3(Q2, A2, p2) * rs).sum()

        out = torch.empty(_n_ext(p), dtype=torch.float64, device=self.dev)
        for e in range(_n_ext(p)):
            v = point(e)
            out[e] = v.detach()
            if grad_out is not None:
                (v * grad_out[e]).backward()
        return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "serve" or c["kind"].startswith("flow"):
        return None
    p, tables, rng = _inputs(c, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = torch.tensor(tables, device=dev, requires_grad=c["kind"] == "d4grad")
    x = _Exact(p, t, c["k"], dev)
    if c["kind"] == "d4grad":
        out = x.d4(torch.tensor(rng.uniform(-1.0, 1.0, _n_ext(p)), device=dev))
        return {"out": out, "grad": t.grad}
    if c["kind"] == "states":
        return x.ft(_states(c, p, rng).to(dev))
    return {D3: x.d3, D4: x.d4, D4F: x.d4, FT: x.ft, FT4: x.ft4}[p.model]()
