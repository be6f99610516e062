"""Rounding of the stencils on fields that vary slowly, where the differences are
small against the values: element by element within a few units in the last place
of the terms of the factored form, whose differences of neighbouring values are
exact there.  The reference is evaluated in extended precision."""
import numpy as np
import pytest

import mfg_inputs as mi

from _gpu_helpers import dev, host, lib

pytestmark = pytest.mark.gpu

LD, U = np.longdouble, 2.0 ** -53
BCS = [("periodic", "periodic"), ("neumann", "periodic"), ("neumann", "neumann")]


def _problem(nx, ny, nt, bc, length, nu):
    return dict(mi.small(seed=1, dim=2, nx=nx, ny=ny, nt=nt, bc=bc, nu=nu)["problem"], len=length)


def _field(nx, ny, nt, seed, slow=1.0):
    """3 plus low modes of amplitude about 1/2, periodic on the node lattice."""
    rng = np.random.Generator(np.random.PCG64(seed))
    X, Y = np.meshgrid(2 * np.pi * np.arange(nx) / nx, 2 * np.pi * np.arange(ny) / ny, indexing="ij")
    t = (np.arange(nt) / nt).reshape(nt, 1, 1)
    a, b = rng.uniform(0, 6, 2)
    return 3.0 + 0.3 * np.cos(X + a)[None] * np.cos(slow * t + b) + 0.2 * np.sin(Y + X + b)[None] * np.cos(slow * t + a)


class _Nb:
    """Neighbour differences of an extended-precision field (0 across a Neumann end)."""

    def __init__(self, p):
        self.per = [b == "periodic" for b in p["bc"]]
        h = [LD(l) / (n if q else n + 1) for l, n, q in zip(p["len"], p["n"], self.per)]
        self.ih, self.nu, self.idt = [1 / v for v in h], LD(p["nu"]), LD(p["nt"]) / LD(p["T"])

    def fwd(self, a, ax):  # a_{i+1} - a_i
        d = np.roll(a, -1, 1 + ax) - a
        if not self.per[ax]:
            d[(slice(None),) * (1 + ax) + (-1,)] = 0
        return d

    def bwd(self, a, ax):  # a_i - a_{i-1}
        d = a - np.roll(a, 1, 1 + ax)
        if not self.per[ax]:
            d[(slice(None),) * (1 + ax) + (0,)] = 0
        return d

    def K(self, a):
        return sum(self.ih[x] ** 2 * (self.bwd(a, x) - self.fwd(a, x)) for x in range(2))

    def Kabs(self, a):  # the terms of K a by magnitude
        b, out = np.abs(a), 0
        for x in range(2):
            for s in (1, -1):
                out = out + self.ih[x] ** 2 * (b + np.roll(b, s, 1 + x))
        return out

    @staticmethod
    def next(a):
        return np.concatenate([a[1:], np.zeros_like(a[:1])])

    @staticmethod
    def prev(a):
        return np.concatenate([np.zeros_like(a[:1]), a[:-1]])


@pytest.mark.parametrize("ny", [8, 40])
@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("length", [(4.0, 4.0), (4.0, 3.0), (1.0, 5.0)])
def test_AAt_slow_in_time(ny, bc, length):
    """1/dt^2 far above 1/dx^2.  Roundings on the longest path: 4 (u), 2 (X), 7 (q), and
    3 in the coefficients."""
    import torch
    p = _problem(8, ny, 256, bc, length, 0.01)
    f = _field(8, ny, 256, 2, 0.3)
    q = torch.empty(f.size, dtype=torch.float64, device="cuda")
    lib().mfg_apply_AAt(lib().mfg_plan(p), 0, dev(f), q)
    g, a = _Nb(p), f.astype(LD)
    x = g.nu * g.K(a) + (a - g.next(a)) * g.idt
    ref = g.nu * g.K(x) + (x - g.prev(x)) * g.idt + 2 * g.K(a)
    xa = g.nu * g.Kabs(a) + np.abs(a - g.next(a)) * g.idt
    terms = g.nu * g.Kabs(xa) + (xa + g.prev(xa)) * g.idt + 2 * g.Kabs(a)
    assert (np.abs(host(q).reshape(f.shape) - ref) <= 16 * U * terms).all()


@pytest.mark.parametrize("shape,bc", [((33, 64, 3), BCS[0]), ((64, 90, 3), BCS[2]), ((300, 40, 2), BCS[1]),
                                      ((60, 22, 2), BCS[2]), ((60, 21, 2), BCS[0]), ((9, 65, 2), BCS[1])])  # in strips from 22 of 32 lanes on
def test_Ct_slow_in_space(shape, bc):
    """The m row of C^T p: nu K p from exact differences of neighbours.  Roundings: a second
    difference, its scale and sum per axis, the time part, and 3 in each coefficient."""
    import torch
    nx, ny, nt = shape
    p = _problem(nx, ny, nt, bc, (0.7, 0.9), 1.0)
    f = _field(nx, ny, nt, 3, 1e-3)
    x = torch.empty(5 * f.size, dtype=torch.float64, device="cuda")
    lib().mfg_apply_Ct(lib().mfg_plan(p), 0, dev(f), x)
    g, a = _Nb(p), f.astype(LD)
    dt = (a - g.next(a)) * g.idt
    kx, ky = (g.ih[q] ** 2 * (g.bwd(a, q) - g.fwd(a, q)) for q in range(2))
    ref = g.nu * (kx + ky) + dt
    bound = 8 * U * (g.nu * (np.abs(kx) + np.abs(ky)) + np.abs(dt))
    assert (np.abs(host(x)[:f.size].reshape(f.shape) - ref) <= bound).all()


@pytest.mark.parametrize("shape,bc", [((33, 64, 3), BCS[0]), ((64, 90, 3), BCS[2]), ((70, 40, 2), BCS[1]), ((50, 9, 3), BCS[2]),
                                       ((60, 28, 2), BCS[0]), ((60, 27, 2), BCS[1])])  # in strips from 28 of 32 lanes on
@pytest.mark.parametrize("length", [(1.0, 1.0), (0.7, 0.9)])
@pytest.mark.parametrize("nu", [0.0, 1e-3])
def test_C_slow_fluxes(shape, bc, length, nu):
    """div_h w from exact differences of each flux, both of an axis nonzero.  Roundings on
    the longest path: 7 in the sums, 5 in the coefficients."""
    import torch
    nx, ny, nt = shape
    p = _problem(nx, ny, nt, bc, length, nu)
    v = np.stack([_field(nx, ny, nt, 4 + q, 1e-3) * (1.0 if q % 2 or q == 0 else -0.4) for q in range(5)])
    r = torch.empty(v[0].size, dtype=torch.float64, device="cuda")
    lib().mfg_apply_C(lib().mfg_plan(p), 0, dev(v), r)
    g, a = _Nb(p), v.astype(LD)
    dm = (a[0] - g.prev(a[0])) * g.idt
    ref, terms = g.nu * g.K(a[0]) + dm, g.nu * g.Kabs(a[0]) + np.abs(dm)
    for ax in range(2):
        w1, w2 = a[1 + 2 * ax].copy(), a[2 + 2 * ax].copy()
        if not g.per[ax]:  # slots past the ends
            w1[(slice(None),) * (1 + ax) + (-1,)] = 0
            w2[(slice(None),) * (1 + ax) + (0,)] = 0
        d1, d2 = w1 - np.roll(w1, 1, 1 + ax), np.roll(w2, -1, 1 + ax) - w2
        ref = ref + g.ih[ax] * (d1 + d2)
        terms = terms + g.ih[ax] * (np.abs(d1) + np.abs(d2))
    assert (np.abs(host(r).reshape(a[0].shape) - ref) <= 12 * U * terms).all()
