"""The work that users of this library have it do, as measurable cases.

Every case goes through the public binding (the names of include/mfg.h): the
Chambolle-Pock solve, the operators it is made of (the AAt apply, the
constraint and its transpose, the preconditioner, the proximal step), the
gradient by implicit differentiation.  Grids are those of the paper's experiments, of the
benchmark and of the tests (a 1-D torus, 128^2 x 64 tori, the 512^2 x 128 Neumann
square, grids whose axes are no powers of two); `draw` spreads sizes, boundary
conditions, precisions and options over the same ranges.

Inputs come from the seed alone and are made on the GPU: Gaussian-mixture
densities, Fourier or cosine potentials, adjoint states and residuals of mixed
smoothness.  `exact` evaluates the same mathematics with plain torch in
64 bits: dense orthonormal transforms, tridiagonal elimination in time per
spatial mode, bisection for the proximal map.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_01958_gb300 as pkg

PERIODIC, NEUMANN = "periodic", "neumann"
MIXED = ("mixed", "mixed_df", "mixed_tc")
DEV = "cuda"
F64 = torch.float64


def _case(op, nx, ny, nt, bc, precision, name=None, **kw):
    """bc: one letter per axis, p(eriodic) or n(eumann); ny = 1 is the 1-D problem."""
    c = {"op": op, "nx": nx, "ny": ny, "nt": nt, "bc": bc, "precision": precision, "l": 1, "nu": 1e-2,
         "qprime": 2.0, "field": False, "tune": False, "iters": 0, "batch": 1, "cg_tol": 1e-10, "f_b": 0.0}
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # a 1-D torus solve in the binding's default precision: the smallest
        # call, every kernel in it a few microseconds
        _case("solve", 64, 1, 32, "pp", "fp64", "solve_torus_1d", nu=0.1, iters=20),
        # four viscosities of the 128^2 x 64 torus in one plan, launch choices
        # tuned: the paper's viscosity study
        _case("solve", 128, 128, 64, "pp", "mixed_tc", "solve_torus_batch", iters=10, batch=4, tune=True),
        # the first iterations of the large Neumann square (the benchmark's workload)
        _case("solve", 512, 512, 128, "nn", "mixed_tc", "solve_neumann_large", iters=6, tune=True),
        # the dominant operator on its own, at that size
        _case("aat", 512, 512, 128, "nn", "mixed", "aat_large"),
        # the operators of the optimality conditions (C y, C^T z, AAt z) on a ragged grid:
        # what a residual check after a solve evaluates
        _case("operators", 201, 147, 50, "np", "fp64", "operators_ragged"),
        # P^{-1} on a grid of round numbers, no power of two among them, FP32 inside
        _case("precond", 200, 150, 60, "pn", "mixed", "precond_ragged"),
        # P^{-1} in the default precision, DST-I in time
        _case("precond", 256, 256, 64, "nn", "fp64", "precond_fp64", l=2),
        # P^{-1} at the benchmark's size and precision
        _case("precond", 512, 512, 128, "nn", "mixed_tc", "precond_large", tune=True),
        # P^{-1} with a viscosity field nu(x): banded solves per time frequency
        _case("precond", 96, 64, 32, "nn", "mixed", "precond_field", field=True),
        # the primal step (lift, prox, extrapolation) at a size between the workloads
        _case("prox_step", 256, 256, 128, "pp", "mixed", "prox_step"),
        # the proximal map of a power Hamiltonian |p|^q'/q' and a quadratic coupling
        _case("prox", 120, 96, 40, "nn", "fp64", "prox_power", qprime=1.5, f_b=0.5),
        # gradients of a terminal loss by implicit differentiation
        _case("adjoint", 128, 128, 64, "pp", "mixed", "adjoint_torus", nu=0.05),
    ]


def draw(rng):
    """One more case of the listed ranges: sizes over their logarithm, odd ones
    among them, every direction, precision and option in turn."""
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        if rng.random() < 0.3:  # powers of two as often as users choose them
            n = 1 << max(3, int(round(math.log2(n))))
        return max(lo, min(hi, n))

    op = rng.choice(["solve", "solve", "aat", "operators", "precond", "precond", "precond", "prox_step", "prox", "adjoint"])
    dim = 1 if rng.random() < 0.15 else 2
    cap = {"solve": 1 << 20, "adjoint": 1 << 18, "prox": 1 << 20, "aat": 1 << 25}.get(op, 1 << 23)
    for _ in range(1000):
        nx = size(8, 512)
        ny = 1 if dim == 1 else size(8, 512)
        nt = size(8, 200)
        if nx * ny * nt <= cap:
            break
    bc = rng.choice("pn") + rng.choice("pn")
    precision = rng.choice(["fp64", "mixed", "mixed", "mixed_tc", "mixed_df"])
    c = _case(op, nx, ny, nt, bc, precision, l=rng.choice([1, 1, 1, 2]), nu=round(10.0 ** rng.uniform(-3, 0), 4))
    if op == "solve":
        c["iters"] = rng.randint(2, 10)
        c["batch"] = rng.choice([1, 1, 2, 3]) if nx * ny * nt <= 1 << 18 else 1
        c["tune"] = rng.random() < 0.5
    if op == "adjoint":
        c["nu"] = round(10.0 ** rng.uniform(-1.5, 0), 4)
    if op in ("prox", "prox_step"):
        c["qprime"] = rng.choice([2.0, 2.0, 1.5, 3.0]) if nx * ny * nt <= 1 << 18 else 2.0
        c["f_b"] = rng.choice([0.0, 0.0, 0.5])
    if op == "precond" and rng.random() < 0.2:
        c.update(field=True, nx=size(8, 64), ny=1 if dim == 1 else size(8, 64), nt=size(8, 48))
    return c


# ----------------------------------------------------------------- inputs --
def _shape(case):
    return case["nt"], case["nx"], case["ny"]


def _dim(case):
    return 1 if case["ny"] == 1 else 2


def _planes(case):
    return 1 + 2 * _dim(case)


def _bcs(case):
    b = [PERIODIC if ch == "p" else NEUMANN for ch in case["bc"]]
    return (b[0], PERIODIC if _dim(case) == 1 else b[1])


def _spacing(case):
    n = (case["nx"], case["ny"])
    return [1.0 / n[a] if _bcs(case)[a] == PERIODIC else 1.0 / (n[a] + 1) for a in range(2)]


def _nus(case):
    """The viscosities of a batch: the case's own and ten times more each."""
    return [min(1.0, case["nu"] * 10.0 ** b / (10.0 if case["batch"] > 2 else 1.0)) for b in range(case["batch"])]


def _nodes(case):
    dx = _spacing(case)
    ax = [torch.arange(n, dtype=F64, device=DEV) + (0 if b == PERIODIC else 1)
          for n, b in zip((case["nx"], case["ny"]), _bcs(case))]
    return torch.meshgrid(ax[0] * dx[0], ax[1] * (dx[1] if _dim(case) == 2 else 0.0), indexing="ij")


def _density(case, rng, floor=0.0):
    """A normalised mixture of three Gaussians (nearest periodic image)."""
    X, Y = _nodes(case)
    m = torch.full_like(X, floor)
    for _ in range(3):
        s = rng.uniform(0.05, 0.15)
        d2 = torch.zeros_like(X)
        for a, P in enumerate((X, Y)[: _dim(case)]):
            d = P - rng.uniform(0.0, 1.0)
            if _bcs(case)[a] == PERIODIC:
                d = d - torch.round(d)
            d2 += d * d
        m += torch.exp(-d2 / (2 * s * s))
    return m / m.mean()


def _potential(case, rng, std=0.5):
    """Eight low modes: Fourier on the torus, cosine series on a Neumann square."""
    X, Y = _nodes(case)
    V = torch.zeros_like(X)
    for _ in range(8):
        k = rng.integers(0, 4, size=2)
        t = [math.pi * (2 if b == PERIODIC else 1) * float(q) for q, b in zip(k, _bcs(case))]
        ph = [rng.uniform(0, 2 * math.pi) if b == PERIODIC else 0.0 for b in _bcs(case)]
        V += rng.normal(0.0, std) / (1.0 + float(k @ k)) * torch.cos(t[0] * X + ph[0]) * torch.cos(t[1] * Y + ph[1])
    return V


def _noise(shape, rng):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(rng.integers(1 << 31)))
    return torch.randn(shape, dtype=F64, device=DEV, generator=g)


def _dual(case, rng, noise):
    """A space-time multiplier: low modes drifting in time, plus noise."""
    nt = case["nt"]
    t = (torch.arange(nt, dtype=F64, device=DEV) / nt).reshape(nt, 1, 1)
    z = torch.zeros(_shape(case), dtype=F64, device=DEV)
    for _ in range(3):
        z += _potential(case, rng, 0.3)[None] * torch.cos(math.pi * rng.uniform(0.0, 3.0) * t + rng.uniform(0.0, 3.0))
    if noise:
        z += noise * _noise(z.shape, rng)
    return z


def _primal(case, rng, floor):
    """(m, w): one mixture flowing into another, w = m v with v in the cone K;
    with floor = 0 cells far from the mass are empty."""
    nt = case["nt"]
    a, b = _density(case, rng, floor), _density(case, rng, floor)
    t = (torch.arange(1, nt + 1, dtype=F64, device=DEV) / nt).reshape(nt, 1, 1)
    m = (1 - t) * a[None] + t * b[None]
    if not floor:
        m = torch.where(m > 1e-3, m, torch.zeros_like(m))
    y = [m]
    for q in range(_planes(case) - 1):
        v = _dual(case, rng, 0.0)
        y.append(m * (v.clamp(min=0.0) if q % 2 == 0 else v.clamp(max=0.0)))
    return torch.stack(y)


def _nu_field(case, rng):
    """A smooth viscosity field, 10 : 1 around the case's viscosity."""
    u = _potential(case, rng, 1.0)
    span = float(u.max() - u.min())
    u = 2.0 * (u - u.min()) / span - 1.0 if span > 0 else torch.zeros_like(u)
    return case["nu"] * 10.0 ** (0.5 * u)


def _inputs(case, seed):
    """What the call gets, as tensors on the GPU (a dict), made from the seed alone."""
    rng = np.random.default_rng([int(seed), case["nx"], case["ny"], case["nt"]])
    op = case["op"]
    out = {}
    if op == "solve":
        per = [(_density(case, rng), _potential(case, rng), 0.1 * _density(case, rng)) for _ in range(case["batch"])]
        out["m0"], out["V"], out["W"] = (torch.stack([p[k] for p in per]) for k in range(3))
        y = torch.zeros((case["batch"], _planes(case)) + _shape(case), dtype=F64, device=DEV)
        y[:, 0] = out["m0"][:, None]
        out["y"] = y
    elif op in ("aat", "precond"):
        out["p"] = _dual(case, rng, 0.5)
    elif op == "operators":
        out["z"] = _dual(case, rng, 0.05)
        out["y"] = _primal(case, rng, 0.0)
    elif op in ("prox", "prox_step"):
        out["V"], out["W"] = _potential(case, rng), 0.1 * _density(case, rng)
        out["y"] = _primal(case, rng, 0.0)
        if op == "prox_step":
            out["z"] = _dual(case, rng, 1e-3) * 0.05
        else:
            out["y"] = out["y"] + 0.2 * _noise(out["y"].shape, rng)
    elif op == "adjoint":
        out["y"] = _primal(case, rng, 0.5)
        out["z"] = _dual(case, rng, 0.0)
        out["gy"] = torch.zeros_like(out["y"])
        dx = _spacing(case)
        vol = dx[0] * (dx[1] if _dim(case) == 2 else 1.0)
        out["gy"][0, -1] = 2.0 * vol * (out["y"][0, -1] - _density(case, rng, 0.5))
    if case["field"]:
        out["nu_field"] = _nu_field(case, rng)
    return out


def _problem(case, nu, field=None):
    p = {"dim": _dim(case), "n": (case["nx"], case["ny"]), "len": (1.0, 1.0), "bc": _bcs(case), "nt": case["nt"],
         "T": 1.0, "nu": nu, "qprime": case["qprime"], "f_a": 1.0, "f_b": case["f_b"], "g_a": 0.0, "l": case["l"],
         "gamma": 1e-3, "tau0": 1.0, "sigma0": 1.0, "max_cp": case["iters"], "cp_tol": 0.0, "cg_rule": 0,
         "cg_tol": case["cg_tol"], "max_cg": 10000}
    if field is not None:
        p["nu_field"] = field.cpu().numpy()
    return p


TAU = 0.6  # a primal step size from the middle of a run
ADJ_TOL = 1e-12


def prepare(case, seed):
    L = pkg.lib()
    s = {"case": case, "L": L}
    s.update(_inputs(case, seed))
    s["plan"] = L.mfg_plan([_problem(case, nu, s.get("nu_field")) for nu in _nus(case)], precision=case["precision"])
    if case["tune"]:
        L.mfg_autotune(s["plan"])
    op = case["op"]
    if op == "solve":
        s["y0"] = s["y"].clone()
        s["ybar"] = torch.empty_like(s["y"])
        s["z"] = torch.empty((case["batch"],) + _shape(case), dtype=F64, device=DEV)
    elif op in ("aat", "precond"):
        s["out"] = torch.empty_like(s["p"])
    elif op == "operators":
        s["r"], s["q"], s["x"] = torch.empty_like(s["z"]), torch.empty_like(s["z"]), torch.empty_like(s["y"])
    elif op == "prox":
        s["out"] = torch.empty_like(s["y"])
    elif op == "prox_step":
        s["new"], s["ybar"] = torch.empty_like(s["y"]), torch.empty_like(s["y"])
    elif op == "adjoint":
        s["dm0"], s["dV"], s["dW"] = (torch.empty((case["nx"], case["ny"]), dtype=F64, device=DEV) for _ in range(3))
        s["dnu"] = torch.empty(1, dtype=F64, device=DEV)
    torch.cuda.synchronize()
    return s


def run(s):
    L, plan, op = s["L"], s["plan"], s["case"]["op"]
    if op == "solve":
        # a fresh solve from the initial iterate in the caller's buffers
        s["y"].copy_(s["y0"])
        s["ybar"].copy_(s["y0"])
        s["z"].zero_()
        L.mfg_solve(plan, s["m0"], s["V"], s["W"], s["y"], s["ybar"], s["z"])
        return {"y": s["y"], "ybar": s["ybar"], "z": s["z"]}
    if op == "aat":
        L.mfg_apply_AAt(plan, 0, s["p"], s["out"])
        return s["out"]
    if op == "precond":
        L.mfg_apply_precond(plan, 0, s["p"], s["out"])
        # the mixed precisions compute the apply in FP32: a caller keeps it as such
        return s["out"].to(torch.float32) if s["case"]["precision"] in MIXED else s["out"]
    if op == "operators":
        L.mfg_apply_C(plan, 0, s["y"], s["r"])
        L.mfg_apply_Ct(plan, 0, s["z"], s["x"])
        L.mfg_apply_AAt(plan, 0, s["z"], s["q"])
        return {"r": s["r"], "x": s["x"], "q": s["q"]}
    if op == "prox":
        L.mfg_prox(plan, 0, TAU, s["y"], s["V"], s["W"], s["out"])
        return s["out"]
    if op == "prox_step":
        # the step works in place; the caller keeps the old iterate
        s["new"].copy_(s["y"])
        L.mfg_prox_step(plan, 0, TAU, s["z"], s["new"], s["ybar"], s["V"], s["W"])
        return {"y": s["new"], "ybar": s["ybar"]}
    L.mfg_adjoint(plan, 0, s["y"], s["z"], s["gy"], s["dm0"], s["dV"], s["dW"], s["dnu"], tol=ADJ_TOL)
    return {"dm0": s["dm0"], "dV": s["dV"], "dW": s["dW"], "dnu": s["dnu"]}


def work(case):
    """Bytes: every input read and every output written once (per iteration for
    a solve, whose state is larger than the caches; at least one operator and
    one preconditioner apply in each).  Flops: stencil terms, n log n
    transforms, elimination in time, one evaluation of the prox equation."""
    n, c, op = case["nx"] * case["ny"] * case["nt"], _planes(case), case["op"]
    d = _dim(case)
    aat = (16, 14 + 12 * d)
    pre = (16, 2 * 2.5 * sum(math.log2(k) for k in (case["nx"], case["ny"]) if k > 1) + 9)
    cc = (8 * c + 8, 4 + 6 * d)
    if case["field"]:
        pre = (16, 4 * 2.0 * 2 * max(1, min(case["nx"], case["ny"])) + 9)
    prox = (16 * c, 10 * c + 20)
    if op == "aat":
        b, f = aat
    elif op == "operators":
        b, f = aat[0] + 2 * cc[0], aat[1] + 2 * cc[1]
    elif op == "precond":
        b, f = pre
        if case["precision"] in MIXED:
            b = 12
    elif op == "prox":
        b, f = prox
    elif op == "prox_step":
        b, f = 8 + 24 * c, prox[1] + cc[1] + 2 * c
    elif op == "solve":
        b = case["iters"] * (16 + 32 * c) * case["batch"]
        f = case["iters"] * (aat[1] + pre[1] + cc[1] + prox[1]) * case["batch"]
    else:
        b, f = 16 * c + 8, (aat[1] + pre[1] + 10 * c) * 30
    return {"bytes": float(b * n), "flops": float(f * n)}


# ------------------------------------------------------- the same in 64 bits --
class _Exact:
    """Plain torch evaluation of one instance."""

    def __init__(self, case, nu):
        self.c, self.nu, self.nt = case, nu, case["nt"]
        self.idt = float(self.nt)
        self.d = _dim(case)
        self.dx = _spacing(case)
        self.per = [b == PERIODIC for b in _bcs(case)]

    def fwd(self, a, ax):
        """a at the plus neighbour minus a, 0 past a Neumann end (axis 0 = x, 1 = y)."""
        k = a.dim() - 2 + ax
        f = torch.roll(a, -1, k) - a
        if not self.per[ax]:
            f.select(k, f.shape[k] - 1).zero_()
        return f

    def back(self, f, ax):
        """The face values f minus those of the minus face (the transpose of -fwd)."""
        k = f.dim() - 2 + ax
        if self.per[ax]:
            return f - torch.roll(f, 1, k)
        g = f.clone()
        g.select(k, g.shape[k] - 1).zero_()
        h = torch.roll(g, 1, k)
        h.select(k, 0).zero_()
        return g - h

    def K(self, a):
        out = torch.zeros_like(a)
        for ax in range(self.d):
            out -= self.back(self.fwd(a, ax), ax) / self.dx[ax] ** 2
        return out

    def C(self, y):
        """Row k: (nu K + I/dt) m^{k+1} - m^k/dt + div_h w^k, the m0 term left out."""
        m = y[0]
        r = self.nu * self.K(m) + self.idt * m
        r[1:] -= self.idt * m[:-1]
        for ax in range(self.d):
            k = m.dim() - 2 + ax
            w1, w2 = y[1 + 2 * ax], y[2 + 2 * ax]
            flux = w1 + torch.roll(w2, -1, k)  # face (i, i+1): w1_i + w2_{i+1}
            if not self.per[ax]:
                flux.select(k, flux.shape[k] - 1).zero_()
            r += self.back(flux, ax) / self.dx[ax]
        return r

    def Ct(self, p):
        x = [self.nu * self.K(p) + self.idt * p]
        x[0][:-1] -= self.idt * p[1:]
        for ax in range(self.d):
            k = p.dim() - 2 + ax
            g = -self.fwd(p, ax) / self.dx[ax]
            h = torch.roll(g, 1, k)
            if not self.per[ax]:
                h.select(k, 0).zero_()
            x += [g, h]
        return torch.stack(x)

    def _axis(self, ax):
        n = (self.c["nx"], self.c["ny"])[ax]
        a = torch.arange(n, dtype=F64, device=DEV)
        if self.per[ax]:
            th = 2 * math.pi * torch.remainder(a[:, None] * a[None], n) / n
            return (torch.cos(th) + torch.sin(th)) / math.sqrt(n), 2 - 2 * torch.cos(2 * math.pi * a / n)
        H = torch.cos(math.pi * a[:, None] * (2 * a[None] + 1) / (2 * n)) * math.sqrt(2.0 / n)
        H[0] = math.sqrt(1.0 / n)
        return H, 2 - 2 * torch.cos(math.pi * a / n)

    def bases(self):
        if not hasattr(self, "H"):
            self.H, lam = zip(*(self._axis(a) for a in range(2)))
            kap = lam[0][:, None] / self.dx[0] ** 2
            self.kap = kap + lam[1][None] / self.dx[1] ** 2 if self.d == 2 else kap
        return self.H

    def modal(self, r, corner):
        """(block tridiagonal in time)^{-1} r, mode by mode: diagonal
        L^2 + 2 kappa + 1/dt^2 and off-diagonal -L/dt for AAt (corner None: first entry
        without 1/dt^2); for P diagonal nu^2 kappa^2 + 2 kappa + 2 L/dt with the
        first entry's 2 L/dt times corner."""
        Hx, Hy = self.bases()
        v = torch.matmul(torch.matmul(Hx, r), Hy.T)
        L = self.nu * self.kap + self.idt
        off = L * self.idt
        if corner is None:
            d0, d1 = L * L + 2 * self.kap, L * L + 2 * self.kap + self.idt ** 2
        else:
            base = self.nu ** 2 * self.kap ** 2 + 2 * self.kap
            d0, d1 = base + corner * off, base + 2 * off
        den, prev = [], None
        for k in range(self.nt):
            den.append(d0 if k == 0 else d1 - off * off / den[-1])
            v[k] = v[k] if k == 0 else v[k] + off / den[-2] * v[k - 1]
        for k in range(self.nt - 1, -1, -1):
            v[k] = (v[k] if k == self.nt - 1 else v[k] + off * v[k + 1]) / den[k]
        return torch.matmul(torch.matmul(Hx.T, v), Hy)

    def precond(self, r, l):
        # the second difference of DCT-VIII (l = 1) has 1 as its first entry, that of DST-I 2
        return self.modal(r.clone(), float(l))

    def precond_field(self, r, l, field):
        """Dense factorisations of (K_nu^2 + 2 K + lambda_k (K_nu + I/dt)/dt)."""
        nx, ny, nt = self.c["nx"], self.c["ny"], self.nt
        S = nx * ny
        eye = torch.eye(S, dtype=F64, device=DEV).reshape(S, nx, ny)
        Kn, K = torch.zeros_like(eye), self.K(eye)
        for ax in range(self.d):
            nf = 0.5 * (field + torch.roll(field, -1, ax)) / self.dx[ax] ** 2
            Kn -= self.back(nf[None] * self.fwd(eye, ax), ax)
        Kn, K, eye = (a.reshape(S, S) for a in (Kn, K, eye))
        chat = Kn @ Kn + 2 * K
        lhat = (Kn + self.idt * eye) * self.idt
        j = torch.arange(nt, dtype=F64, device=DEV)
        if l == 1:
            lam = 2 - 2 * torch.cos(math.pi * (j + 0.5) / (nt + 0.5))
            V = 2 / math.sqrt(2 * nt + 1) * torch.cos(math.pi * (2 * j[:, None] + 1) * (2 * j[None] + 1) / (2 * (2 * nt + 1)))
        else:
            lam = 2 - 2 * torch.cos(math.pi * (j + 1) / (nt + 1))
            V = math.sqrt(2 / (nt + 1)) * torch.sin(math.pi * (j[:, None] + 1) * (j[None] + 1) / (nt + 1))
        b = V @ r.reshape(nt, S)
        for k in range(nt):
            b[k] = torch.cholesky_solve(b[k][:, None], torch.linalg.cholesky(chat + lam[k] * lhat))[:, 0]
        return (V @ b).reshape(r.shape)

    def prox(self, tau, v, V, W):
        """Per cell and per plane: bisection of the increasing equation for m."""
        q = self.c["qprime"] / (self.c["qprime"] - 1.0)
        out = torch.empty_like(v)
        step = max(1, (1 << 22) // V.numel())
        for k0 in range(0, self.nt, step):
            vv = v[:, k0:k0 + step]
            c = V[None].expand(vv.shape[1:]).clone()
            if k0 + step >= self.nt:
                c[-1] += W * self.idt
            P = torch.stack([vv[i].clamp(min=0.0) if i % 2 else vv[i].clamp(max=0.0) for i in range(1, v.shape[0])])
            Pn = (P * P).sum(0).sqrt()
            B = vv[0] - tau * c
            a1, tb, qp = 1.0 + tau, tau * self.c["f_b"], self.c["qprime"]

            def speed(m):  # t with m t + tau t^(q-1) = |P|
                if q == 2.0:
                    return Pn / (m + tau)
                lo, hi = torch.zeros_like(Pn), (Pn / tau) ** (1.0 / (q - 1.0))
                for _ in range(64):
                    t = 0.5 * (lo + hi)
                    low = m * t + tau * t ** (q - 1.0) < Pn
                    lo, hi = torch.where(low, t, lo), torch.where(low, hi, t)
                return 0.5 * (lo + hi)

            lim = tau / qp * (Pn / tau) ** qp
            lo, hi = torch.zeros_like(Pn), B.clamp(min=0.0) + lim
            for _ in range(80):
                m = 0.5 * (lo + hi)
                low = a1 * m + tb * m * m - B - tau / qp * speed(m) ** q < 0
                lo, hi = torch.where(low, m, lo), torch.where(low, hi, m)
            m = torch.where(B + lim <= 0, torch.zeros_like(B), 0.5 * (lo + hi))
            s = torch.where((Pn > 0) & (m > 0), m * speed(m) / torch.where(Pn > 0, Pn, torch.ones_like(Pn)), torch.zeros_like(Pn))
            out[0, k0:k0 + step], out[1:, k0:k0 + step] = m, s[None] * P
        return out

    def solve(self, m0, V, W, y, iters):
        tau, sigma = 1.0, 1.0
        ybar, z = y.clone(), torch.zeros_like(y[0])
        for _ in range(iters):
            r = self.C(ybar)
            r[0] -= self.idt * m0
            z = z + self.modal(sigma * r, None)
            new = self.prox(tau, y - tau * self.Ct(z), V, W)
            theta = 1.0 / math.sqrt(1.0 + 2e-3 * tau)
            ybar = new + theta * (new - y)
            y, tau, sigma = new, theta * tau, sigma / theta
        return y, ybar, z

    def adjoint(self, y, z, gy):
        """[mu; eta] of the linearised optimality conditions by conjugate
        gradients on the Schur complement, in 64 bits to round-off."""
        m, w = y[0], y[1:]
        on = m > 0
        im = torch.where(on, 1.0 / torch.where(on, m, torch.ones_like(m)), torch.zeros_like(m))
        act = ((w != 0) & on[None]).to(F64)

        def hinv(u):
            um = torch.where(on, (u[0] + (w * u[1:]).sum(0) * im), torch.zeros_like(m))
            return torch.cat([um[None], act * (m[None] * u[1:] + w * (im * um)[None])])

        r = self.C(hinv(gy))
        stop = 1e-14 * float(r.norm())
        eta = torch.zeros_like(r)
        h = self.precond(r, self.c["l"])
        p, rz = h.clone(), float((r * h).sum())
        for _ in range(3000):
            q = self.C(hinv(self.Ct(p)))
            alpha = rz / float((p * q).sum())
            eta += alpha * p
            r -= alpha * q
            if float(r.norm()) <= stop:
                break
            h = self.precond(r, self.c["l"])
            rz, old = float((r * h).sum()), rz
            p = h + rz / old * p
        mu = hinv(gy - self.Ct(eta))
        dnu = -(mu[0] * self.K(z)).sum() - (eta * self.K(m)).sum()
        return eta[0] * self.idt, -mu[0].sum(0), -mu[0, -1] * self.idt, dnu.reshape(1)


def exact(case, seed):
    s, op = _inputs(case, seed), case["op"]
    E = _Exact(case, case["nu"])
    if op == "aat":
        return E.C(E.Ct(s["p"]))
    if op == "operators":
        return {"r": E.C(s["y"]), "x": E.Ct(s["z"]), "q": E.C(E.Ct(s["z"]))}
    if op == "precond":
        if not case["field"]:
            return E.precond(s["p"], case["l"])
        if case["nx"] * case["ny"] > 6500:
            return None
        return E.precond_field(s["p"], case["l"], s["nu_field"])
    if op == "prox":
        return E.prox(TAU, s["y"], s["V"], s["W"])
    if op == "prox_step":
        new = E.prox(TAU, s["y"] - TAU * E.Ct(s["z"]), s["V"], s["W"])
        return {"y": new, "ybar": new + (new - s["y"]) / math.sqrt(1.0 + 2e-3 * TAU)}
    if op == "solve":
        got = [_Exact(case, nu).solve(s["m0"][b], s["V"][b], s["W"][b], s["y"][b], case["iters"])
               for b, nu in enumerate(_nus(case))]
        return {k: torch.stack([g[i] for g in got]) for i, k in enumerate(("y", "ybar", "z"))}
    if case["nx"] * case["ny"] * case["nt"] > 1 << 21:
        return None
    return dict(zip(("dm0", "dV", "dW", "dnu"), E.adjoint(s["y"], s["z"], s["gy"])))
