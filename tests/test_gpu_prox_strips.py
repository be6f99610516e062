"""The primal step in warp strips: strips with every kind of last lane group, both
boundary conditions, warps whose flux components are all zero, all active and
mixed (the skipped components), an empty density, and tau far from 1, against the
oracle's sparse C^T and bisection prox.

Bars of the existing prox-step test: 1e-12 relative, 1e-11 pointwise."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle import operators as ops
from oracle.prox import prox as oracle_prox

from _gpu_helpers import dev, host, lib, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nt", [(2, 20, 2), (5, 32, 3), (33, 55, 4), (40, 64, 2), (3, 95, 9)])
@pytest.mark.parametrize("bc", [("periodic", "neumann"), ("neumann", "periodic")])
@pytest.mark.parametrize("flux", ["zero", "one-sided", "mixed"])
@pytest.mark.parametrize("tau", [0.01, 0.6, 30.0])
def test_prox_strip(nx, ny, nt, bc, flux, tau):
    import torch
    inst = mi.small(seed=nx * ny, dim=2, nx=nx, ny=ny, nt=nt, bc=bc)
    p = inst["problem"]
    s, n, c = ops.sizes(p)
    y0 = mi.random_field((c, nt, nx, ny), 81, -1.0, 1.0)
    y0[0] = np.maximum(y0[0], 0.0)
    z = mi.random_field(n, 82, -0.5, 0.5)
    if flux == "zero":        # old fluxes zero, z monotone: one direction per axis everywhere inside
        y0[1:] = 0.0
        X, Y = np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij")
        z = (0.01 * X - 0.02 * Y)[None].repeat(nt, 0).reshape(-1)
    elif flux == "one-sided":
        y0[2::2] = 0.0
        y0[1::2] = np.abs(y0[1::2])
    y, ybar = dev(y0), torch.empty(c * n, dtype=torch.float64, device="cuda")
    lib().mfg_prox_step(lib().mfg_plan(p), 0, tau, dev(z), y, ybar, dev(inst["V"]), dev(inst["W"]))
    x = ops.constraint(p).T @ z
    ref = oracle_prox(p, tau, (y0.reshape(-1) - tau * x).reshape(y0.shape), inst["V"], inst["W"]).reshape(-1)
    theta = 1.0 / np.sqrt(1.0 + 2.0 * p["gamma"] * tau)
    ref_bar = ref + theta * (ref - y0.reshape(-1))
    assert rel(host(y), ref) <= 1e-12
    assert np.abs(host(y) - ref).max() <= 1e-11 * max(1.0, np.abs(ref).max())
    assert rel(host(ybar), ref_bar) <= 1e-12
