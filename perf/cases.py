"""The work that users of the solver have it do, as measurable cases.

A case is a dict of plain values.  `kind` says which public entry point a pass goes through:

  solve   Solver.set_rhs(g on the device) and Solver.solve(): a new right-hand side on a kept
          solver, the result left on the device
  host    fmg_set_rhs / fmg_solve with pinned host buffers: the same, end to end from the host
  batch   set_rhs on every instance of a kept Batch, then Batch.solve()
  serve   a burst of requests with host buffers through a kept Server
  vcycle  fmg_vcycle_noalloc: linear V-cycles from zero on a caller's own arrays

Right-hand sides are what the method meets in earnest: g of a manufactured solution (a sum of
seeded sine modes, g = -Laplace(u*) + a f(u*)) or a sum of seeded sine modes itself.  Sizes and
options are those of paper_1611_05677_gb300/workloads.py, the tests and bench.py, and drawn cases
spread over the same ranges (meshes of 2^k cells per side).
"""
import itertools
import math

import numpy as np
import torch

from paper_1611_05677_gb300 import fmg

F_ALL = ("cubic", "expm1", "linear", "signed_pow32", "neg_exp_neg")


def _solve(name, dim, H, r, f, precision, smoother, rhs, kind="solve", a=1.0, p=1, coefficient=False):
    return {"name": name, "kind": kind, "dim": dim, "H": H, "r": r, "f": f, "a": a, "precision": precision,
            "smoother": smoother, "rhs": rhs, "p": p, "coefficient": coefficient}


def listed():
    return [
        # the small 2D problem with the library's default settings: one quick solve, all latency
        _solve("2d_65_fp64", 2, 4, 4, "cubic", "fp64", "rbgs", "manufactured"),
        # a small request of a served mix, solved directly
        _solve("2d_129_mixed", 2, 4, 5, "expm1", "mixed", "chebyshev", "modes"),
        # the odd 3/2 power and the default smoother, a middle size
        _solve("2d_513_mixed_rbgs", 2, 8, 6, "signed_pow32", "mixed", "rbgs", "manufactured"),
        # a diffusion coefficient that jumps between the coarse cells
        _solve("2d_1025_coefficient", 2, 8, 7, "cubic", "mixed", "rbgs", "modes", coefficient=True),
        # the headline problem, 4.19 M unknowns, in both precisions
        _solve("2d_2049_mixed", 2, 8, 8, "cubic", "mixed", "chebyshev", "manufactured"),
        _solve("2d_2049_fp64", 2, 8, 8, "cubic", "fp64", "rbgs", "manufactured"),
        # the cube problem, 16.6 M unknowns
        _solve("3d_257_mixed", 3, 4, 6, "expm1", "mixed", "chebyshev", "manufactured"),
        # the cube one refinement coarser, every step in FP64
        _solve("3d_129_fp64", 3, 4, 5, "expm1", "fp64", "rbgs", "manufactured"),
        # the headline problem from and to pinned host memory, as an application calls it
        _solve("2d_2049_host", 2, 8, 8, "cubic", "mixed", "chebyshev", "manufactured", kind="host"),
        # independent instances of mixed sizes (5 to 8 refinements of 1/H = 4) solved together
        {"name": "batch_32_mixed", "kind": "batch", "count": 32, "rmin": 5, "rmax": 8, "mix": 0, "precision": "mixed",
         "smoother": "chebyshev"},
        # a burst of 2D and 3D requests with host buffers
        {"name": "serve_24_mixed", "kind": "serve", "count": 24, "r2d": 8, "r3d": 5, "mix": 0, "precision": "mixed",
         "smoother": "chebyshev"},
        # linear V-cycles on a caller's arrays where no device memory may be allocated
        {"name": "vcycle_2d_513_fp64", "kind": "vcycle", "dim": 2, "H": 4, "level": 8, "cycles": 4},
    ]


def _log_int(rng, lo, hi):
    """An integer of lo..hi, spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("solve",) * 6 + ("host", "batch", "serve", "vcycle"))
    if kind == "vcycle":
        dim = rng.choice((2, 3))
        H = rng.choice((2, 4, 8)) if dim == 2 else rng.choice((2, 4))
        nmax = 1024 if dim == 2 else 128
        level = rng.randint(4, int(math.log2(nmax / H)) + 1)
        return {"kind": kind, "dim": dim, "H": H, "level": level, "cycles": _log_int(rng, 1, 10)}
    mixed = rng.random() < 0.6
    precision = "mixed" if mixed else "fp64"
    smoother = rng.choice(("chebyshev", "chebyshev", "rbgs")) if mixed else rng.choice(("rbgs", "rbgs", "chebyshev"))
    if kind == "batch":
        rmax = rng.randint(5, 8 if mixed else 7)
        return {"kind": kind, "count": _log_int(rng, 2, 32), "rmin": rng.randint(3, rmax), "rmax": rmax,
                "mix": rng.randint(1, 999), "precision": precision, "smoother": smoother}
    if kind == "serve":
        return {"kind": kind, "count": _log_int(rng, 2, 24), "r2d": rng.randint(5, 8 if mixed else 7),
                "r3d": rng.randint(3, 5 if mixed else 4), "mix": rng.randint(1, 999), "precision": precision,
                "smoother": smoother}
    dim = rng.choice((2, 2, 2, 3)) if kind == "solve" else rng.choice((2, 3))
    H = rng.choice((2, 4, 8)) if dim == 2 else rng.choice((2, 4))
    nmax = 2048 if dim == 2 else 256 if mixed else 128
    rmax = int(math.log2(nmax / H))
    r = rng.randint(3, rmax)
    coefficient = kind == "solve" and rng.random() < 0.15
    return _drawn(_solve("", dim, H, r, rng.choice(F_ALL), precision, "rbgs" if coefficient else smoother,
                         rng.choice(("manufactured", "modes")), kind=kind, a=round(rng.uniform(0.5, 2.0), 3),
                         p=rng.choice((1, 1, 1, 2)) if r < rmax else 1, coefficient=coefficient))


def _drawn(case):
    del case["name"]
    return case


# ------------------------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _modes(rng, dim, uniform):
    """Eight sine modes (frequencies per axis, amplitude), without replacement."""
    kmax = 6 if dim == 2 else 4
    pick = rng.choice(kmax ** dim, size=8, replace=False)
    kv = [np.unravel_index(int(i), (kmax,) * dim) for i in pick]
    amp = rng.uniform(0.0, 1.0, 8) if uniform else rng.standard_normal(8)
    return [([int(k) + 1 for k in ks], float(c)) for ks, c in zip(kv, amp)]


def _mode_sum(modes, dim, n, laplace=False):
    """sum c sin(k1 pi x) sin(k2 pi y) .. on the (n+1)^dim nodes (x last), or of -Laplace of it."""
    dev = _device()
    x = torch.arange(n + 1, dtype=torch.float64) / n
    out = torch.zeros((n + 1,) * dim, dtype=torch.float64, device=dev)
    for ks, c in modes:
        amp = c * math.pi ** 2 * sum(k * k for k in ks) if laplace else c
        t = (amp * torch.sin(ks[0] * math.pi * x)).to(dev)
        for k in ks[1:]:
            s = torch.sin(k * math.pi * x).to(dev)
            t = s.reshape((-1,) + (1,) * t.dim()) * t
        out += t
    return out


def _f(kind, a, u):
    if kind == "cubic":
        return a * u ** 3
    if kind == "expm1":
        return a * torch.expm1(u)
    if kind == "linear":
        return a * u
    if kind == "signed_pow32":
        return a * u * torch.sqrt(torch.abs(u))
    return -a * torch.exp(-u)


def _df(kind, a, u):
    if kind == "cubic":
        return 3 * a * u ** 2
    if kind == "expm1":
        return a * torch.exp(u)
    if kind == "linear":
        return torch.full_like(u, a)
    if kind == "signed_pow32":
        return 1.5 * a * torch.sqrt(torch.abs(u))
    return a * torch.exp(-u)


def _rhs(q, rng):
    """Nodal g of one instance; q: dim, H, r, f, a, rhs."""
    n = q["H"] << q["r"]
    if q["rhs"] == "modes":
        return _mode_sum(_modes(rng, q["dim"], False), q["dim"], n)
    modes = _modes(rng, q["dim"], q["dim"] == 3 or q["f"] != "cubic")
    return _mode_sum(modes, q["dim"], n, laplace=True) + _f(q["f"], q["a"], _mode_sum(modes, q["dim"], n))


def _coefficient(q):
    """The entries of A(x) per coarse cell: a property of the problem, not of the seed."""
    if not q.get("coefficient"):
        return None
    return np.random.default_rng(3).uniform(0.5, 2.0, size=(q["H"] ** q["dim"], q["dim"]))


def _instances(case):
    """The problems of a case; those of a batch or a burst are drawn from its `mix`."""
    if case["kind"] in ("solve", "host"):
        return [case]
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        q = {"H": 4, "rhs": "modes", "p": 1, "precision": case["precision"], "smoother": case["smoother"]}
        if case["kind"] == "batch":
            q.update(dim=2, r=int(rng.integers(case["rmin"], case["rmax"] + 1)), f="cubic", a=float(rng.uniform(0.5, 2.0)))
        else:
            dim = 2 if rng.uniform() < 0.7 else 3
            lo, hi = (5, case["r2d"]) if dim == 2 else (3, case["r3d"])
            q.update(dim=dim, r=int(rng.integers(lo, hi + 1)), f="cubic" if rng.uniform() < 0.5 else "expm1", a=1.0)
        out.append(q)
    return out


def _cycles(q):
    return 2 if q["dim"] == 2 else 3


def _params(q):
    return fmg.make_params(dim=q["dim"], coarse_cells=q["H"], refinements=q["r"], f=q["f"], f_scale=q["a"],
                           m_vcycles=_cycles(q), p_corrections=q["p"], precision=q["precision"],
                           smoother=q["smoother"], coefficient=_coefficient(q))


def _vcycle_rhs(case, rng):
    """b of A u = b: the load vector of a smooth field with some noise, zero on the boundary."""
    n = case["H"] << (case["level"] - 1)
    dim = case["dim"]
    gen = torch.Generator(device=_device()).manual_seed(int(rng.integers(1 << 31)))
    b = _mode_sum(_modes(rng, dim, False), dim, n)
    b += 0.1 * torch.randn(b.shape, dtype=torch.float64, device=b.device, generator=gen)
    b /= float(n) ** dim
    out = torch.zeros_like(b)
    inner = (slice(1, n),) * dim
    out[inner] = b[inner]
    return out


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "vcycle":
        b = _vcycle_rhs(case, rng)
        return {"kind": kind, "case": dict(case), "b": b, "u": torch.zeros_like(b)}
    qs = _instances(case)
    gs = [_rhs(q, rng) for q in qs]
    if kind == "serve":
        return {"kind": kind, "server": fmg.Server(max_inflight=8), "params": [_params(q) for q in qs],
                "g": [g.cpu().pin_memory() for g in gs],
                "u": [torch.empty(g.shape, dtype=torch.float64, pin_memory=True) for g in gs]}
    solvers = [fmg.Solver(_params(q), g) for q, g in zip(qs, gs)]
    if kind == "batch":
        return {"kind": kind, "solvers": solvers, "batch": fmg.Batch(solvers), "g": gs}
    if kind == "host":
        return {"kind": kind, "solver": solvers[0], "g": gs[0].cpu().pin_memory(),
                "u": torch.empty(gs[0].shape, dtype=torch.float64, pin_memory=True)}
    return {"kind": kind, "solver": solvers[0], "g": gs[0]}


def run(state):
    kind = state["kind"]
    if kind == "solve":
        state["solver"].set_rhs(state["g"])
        return {"u": state["solver"].solve()}
    if kind == "host":
        ctx = state["solver"].ctx
        fmg.fmg_set_rhs(ctx, state["g"])
        fmg.fmg_solve(ctx, state["u"])
        return {"u": state["u"]}
    if kind == "batch":
        for s, g in zip(state["solvers"], state["g"]):
            s.set_rhs(g)
        state["batch"].solve()
        return {"u": [s.solution() for s in state["solvers"]]}
    if kind == "serve":
        server = state["server"]
        for p, g, u in zip(state["params"], state["g"], state["u"]):
            server.submit(p, g, u)
        server.drain()
        left = len(state["u"])
        while left:
            for r in server.poll():
                if r.status != fmg.FMG_OK:
                    raise fmg.FMGError(r.status, fmg.fmg_server_last_error())
                left -= 1
        return {"u": state["u"]}
    c = state["case"]
    state["u"].zero_()
    fmg.fmg_vcycle_noalloc(c["dim"], c["H"], c["level"], state["b"], state["u"], cycles=c["cycles"])
    return {"u": state["u"]}


# ------------------------------------------------------------------------------- work

def _cycle_flops(dim, smoother):
    """Operations per top-level node of one V(2,2) cycle, its coarser levels included."""
    stencil = 4 * dim + 2
    smooth = 4 * (stencil + (3 if smoother == "chebyshev" else 0))
    return (smooth + stencil + 2 * 2 ** dim + 2) * 2 ** dim / (2 ** dim - 1)


def work(case):
    if case["kind"] == "vcycle":
        nodes = float(((case["H"] << (case["level"] - 1)) + 1) ** case["dim"])
        return {"bytes": 16 * nodes, "flops": case["cycles"] * nodes * _cycle_flops(case["dim"], "rbgs")}
    nbytes = flops = 0.0
    for q in _instances(case):
        dim = q["dim"]
        nodes = float(((q["H"] << q["r"]) + 1) ** dim)
        # per level and correction step: right-hand side, m cycles, the augmented problem's sums
        # (two Newton passes and the update); the coarser levels add a geometric series
        step = 8 + _cycles(q) * (_cycle_flops(dim, q["smoother"]) + 4 * dim + 3) + (130 if dim == 2 else 220)
        nbytes += 16 * nodes
        flops += q["p"] * nodes * step * 2 ** dim / (2 ** dim - 1)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------- exact
# The method itself (nested meshes, V(2,2) cycles, the correction step of eq. 3.4 and 3.6, the
# full multigrid schedule) written out in plain FP64 torch.

class _Level:
    """A_k of one mesh: the axis stencils of the P1 stiffness, with a weight per mesh edge where
    the coefficient is not the identity."""

    def __init__(self, dim, H, level, coef=None):
        self.dim, self.n = dim, H << (level - 1)
        n = self.n
        self.sigma = 1.0 if dim == 2 else 1.0 / n
        self.weight = 1.0 / float(n) ** dim
        self.edge = None
        dev = _device()
        if coef is not None:
            self.edge = []
            cells = torch.tensor(coef, dtype=torch.float64, device=dev).reshape((H,) * dim + (dim,))
            for ax in range(dim):
                c = cells[..., ax]
                for t in range(dim):
                    c = c.repeat_interleave(n // H, dim=t)
                td = dim - 1 - ax                       # tensor axis of coordinate `ax`
                others = [t for t in range(dim) if t != td]

                def part(down):
                    return c[tuple(slice(None) if t == td else slice(0, n - 1) if t in down else slice(1, n)
                                   for t in range(dim))]

                if dim == 2:
                    w = 0.5 * (part(()) + part(others))
                else:
                    w = (2 * part(()) + 2 * part(others) + part(others[:1]) + part(others[1:])) / 6
                self.edge.append((w.narrow(td, 0, n - 1), w.narrow(td, 1, n - 1)))
        ix = torch.arange(1, n, device=dev)
        parity = sum(ix.reshape((-1,) + (1,) * k) for k in range(dim)) % 2
        self.red = parity == 0
        self.diag = 2.0 * dim * self.sigma if self.edge is None else self.sigma * sum(a + b for a, b in self.edge)

    def inner(self, u):
        return u[(Ellipsis,) + (slice(1, self.n),) * self.dim]

    def neighbours(self, u):
        """Sum of the (weighted) axis neighbours at the interior nodes."""
        n, tot = self.n, 0.0
        for ax in range(self.dim):
            td = self.dim - 1 - ax
            lo, hi = (u[(Ellipsis,) + tuple(slice(1 + s, n + s) if t == td else slice(1, n) for t in range(self.dim))]
                      for s in (-1, 1))
            tot = tot + (lo + hi if self.edge is None else self.edge[ax][0] * lo + self.edge[ax][1] * hi)
        return tot

    def apply(self, u):
        out = torch.zeros_like(u)
        self.inner(out).copy_(self.diag * self.inner(u) - self.sigma * self.neighbours(u))
        return out

    def prolong(self, c):
        """The coarse P1 function c at this level's nodes."""
        n, m = self.n, self.n // 2
        out = torch.zeros(c.shape[:c.dim() - self.dim] + (n + 1,) * self.dim, dtype=c.dtype, device=c.device)
        for p in itertools.product((0, 1), repeat=self.dim):
            to = (Ellipsis,) + tuple(slice(k, n + 1 - k, 2) for k in p)
            lo = c[(Ellipsis,) + tuple(slice(0, m + 1 - k) for k in p)]
            hi = c[(Ellipsis,) + tuple(slice(k, m + 1) for k in p)]
            out[to] = 0.5 * (lo + hi)
        return out

    def restrict(self, r):
        """P^T r on the next coarser mesh (zero on its boundary)."""
        n, m = self.n, self.n // 2
        out = torch.zeros(r.shape[:r.dim() - self.dim] + (m + 1,) * self.dim, dtype=r.dtype, device=r.device)
        to = out[(Ellipsis,) + (slice(1, m),) * self.dim]
        for p in itertools.product((0, 1), repeat=self.dim):
            for s in ((1, -1) if any(p) else (1,)):
                at = (Ellipsis,) + tuple(slice(2 + s * k, n - 1 + s * k, 2) for k in p)
                to += (0.5 if any(p) else 1.0) * r[at]
        return out


def _dense(level):
    """A_1 as a dense matrix over the interior nodes."""
    m = (level.n - 1) ** level.dim
    e = torch.eye(m, dtype=torch.float64, device=_device()).reshape((m,) + (level.n - 1,) * level.dim)
    u = torch.zeros((m,) + (level.n + 1,) * level.dim, dtype=torch.float64, device=e.device)
    level.inner(u).copy_(e)
    return torch.stack([level.inner(level.apply(x)).reshape(-1) for x in u])


def _smooth(level, u, b, smoother, steps, post):
    if smoother == "rbgs":
        for _ in range(steps):
            for colour in ((False, True) if post else (True, False)):
                new = (level.inner(b) + level.sigma * level.neighbours(u)) / level.diag
                inner = level.inner(u)
                inner.copy_(torch.where(level.red == colour, new, inner))
        return
    theta, delta = 1.25, 0.75   # the interval [1/2, 2] of D^{-1} A
    rho, d = delta / theta, 0.0
    for k in range(steps):
        z = (level.inner(b) + level.sigma * level.neighbours(u)) / level.diag - level.inner(u)
        if k == 0:
            d = z / theta
        else:
            new = 1.0 / (2.0 * theta / delta - rho)
            d = new * rho * d + 2.0 * new / delta * z
            rho = new
        level.inner(u).add_(d)


def _vcycle(levels, k, u, b, smoother, A1):
    level = levels[k]
    if k == 0:
        level.inner(u).copy_(torch.linalg.solve(A1, level.inner(b).reshape(-1)).reshape(level.inner(u).shape))
        return
    _smooth(level, u, b, smoother, 2, False)
    rc = level.restrict(b - level.apply(u))
    e = torch.zeros_like(rc)
    _vcycle(levels, k - 1, e, rc, smoother, A1)
    u += level.prolong(e)
    _smooth(level, u, b, smoother, 2, True)


def _newton(residual, jacobian, y):
    for _ in range(40):
        step = torch.linalg.solve(jacobian(y), residual(y))
        y = y - step
        if float(step.abs().max()) <= 1e-13 * max(1.0, float(y.abs().max())):
            break
    return y


def _augmented(levels, k, u, g, q, A1):
    """The semilinear problem on V_H + span{u~} (eq. 3.6): alpha u~ + P c."""
    level, dim, kind, a = levels[k], q["dim"], q["f"], q["a"]
    N = A1.shape[0]
    P = torch.zeros((N,) + (levels[0].n + 1,) * dim, dtype=torch.float64, device=u.device)
    levels[0].inner(P).copy_(torch.eye(N, dtype=torch.float64, device=u.device).reshape((N,) + (levels[0].n - 1,) * dim))
    for j in range(1, k + 1):
        P = levels[j].prolong(P)
    B = torch.cat((P, u[None])).reshape(N + 1, -1)
    del P
    mask = torch.zeros_like(u)
    level.inner(mask).fill_(level.weight)
    w = mask.reshape(-1)
    Au = level.apply(u).reshape(-1)
    K = torch.zeros((N + 1, N + 1), dtype=torch.float64, device=u.device)
    K[:N, :N] = A1
    K[N] = B @ Au
    K[:N, N] = K[N, :N]
    gv = g.reshape(-1)

    def residual(y):
        return K @ y + B @ (w * (_f(kind, a, y @ B) - gv))

    def jacobian(y):
        wd = w * _df(kind, a, y @ B)
        J = K.clone()
        for at in range(0, B.shape[1], 1 << 21):
            part = B[:, at:at + (1 << 21)]
            J += (part * wd[at:at + (1 << 21)]) @ part.T
        return J

    y = torch.zeros(N + 1, dtype=torch.float64, device=u.device)
    y[N] = 1.0
    return (_newton(residual, jacobian, y) @ B).reshape(u.shape)


def _full_multigrid(q, g):
    dim, H, r = q["dim"], q["H"], q["r"]
    levels = [_Level(dim, H, k + 1, _coefficient(q)) for k in range(r + 1)]
    gs = [g[(slice(None, None, 1 << (r - k)),) * dim].clone() for k in range(r + 1)]
    A1 = _dense(levels[0])
    first = levels[0]
    g1 = first.inner(gs[0]).reshape(-1)
    y = _newton(lambda y: A1 @ y + first.weight * (_f(q["f"], q["a"], y) - g1),
                lambda y: A1 + first.weight * torch.diag(_df(q["f"], q["a"], y)), torch.zeros_like(g1))
    u = torch.zeros_like(gs[0])
    first.inner(u).copy_(y.reshape(first.inner(u).shape))
    for k in range(1, r + 1):
        u = levels[k].prolong(u)
        for _ in range(q["p"]):
            b = torch.zeros_like(u)
            levels[k].inner(b).copy_(levels[k].inner(levels[k].weight * (gs[k] - _f(q["f"], q["a"], u))))
            for _ in range(_cycles(q)):
                _vcycle(levels, k, u, b, q["smoother"], A1)
            u = _augmented(levels, k, u, gs[k], q, A1)
    return u


def exact(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "vcycle":
        b = _vcycle_rhs(case, rng)
        levels = [_Level(case["dim"], case["H"], k + 1) for k in range(case["level"])]
        A1, u = _dense(levels[0]), torch.zeros_like(b)
        for _ in range(case["cycles"]):
            _vcycle(levels, case["level"] - 1, u, b, "rbgs", A1)
        return {"u": u}
    qs = _instances(case)
    gs = [_rhs(q, rng) for q in qs]
    us = [_full_multigrid(q, g) for q, g in zip(qs, gs)]
    return {"u": us[0]} if case["kind"] in ("solve", "host") else {"u": us}
