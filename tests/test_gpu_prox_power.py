"""The proximal map of the power Hamiltonian |p|^q'/q' over its exponents and
over the cells where the paired FP32 / FP64 root iteration can go wrong (no
flux, vanishing density at the threshold of the zero branch, density or flux
dominating by orders of magnitude, data outside the FP32 range), against the
oracle's nested bisection.

Tolerance: both sides stop at the rounding of the FP64 residuals, a few ulps of
the larger terms; the existing bar of the general map (1e-12 of the largest
value) is kept."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle.prox import prox as oracle_prox

from _gpu_helpers import dev, host, lib

pytestmark = pytest.mark.gpu


def _cells(p, tau, qp, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    shp = (5, p["nt"]) + tuple(p["n"])
    v = rng.uniform(-2.0, 2.0, size=shp)
    k = rng.integers(0, 6, size=shp[1:])
    v[1:] = np.where(k == 1, 0.0, v[1:])                       # no flux
    v[1:] = np.where(k == 2, v[1:] * 1e-6, v[1:])              # density dominates
    v[0] = np.where(k == 3, v[0] * 1e-4, v[0])                 # flux dominates
    P = np.where(np.arange(4).reshape(4, 1, 1, 1) % 2 == 0, np.maximum(v[1:], 0), np.minimum(v[1:], 0))
    lim = (tau / qp) * (np.sqrt((P * P).sum(0)) / tau) ** qp
    near = -lim * (1.0 + rng.choice([-1e-3, -1e-6, 1e-6, 1e-3], size=lim.shape))
    v[0] = np.where(k == 4, near, v[0])                        # the zero branch's threshold (V = W = 0)
    return v


@pytest.mark.parametrize("qp", [1.25, 4.0 / 3.0, 1.5, 1.9, 2.5, 3.0, 5.0])
@pytest.mark.parametrize("f_b", [0.0, 0.5])
def test_power_prox_cells(qp, f_b):
    import torch
    L = lib()
    p = dict(mi.small(seed=7, dim=2, nx=7, ny=11, nt=3, bc=("neumann", "periodic"))["problem"], qprime=qp, f_b=f_b)
    zero = np.zeros(p["n"])
    for tau in (0.05, 6.0):
        v = _cells(p, tau, qp, 17)
        y = torch.empty(v.size, dtype=torch.float64, device="cuda")
        L.mfg_prox(L.mfg_plan(p), 0, tau, dev(v), dev(zero), dev(zero), y)
        ref = oracle_prox(p, tau, v, zero, zero).reshape(-1)
        assert np.abs(host(y) - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())


def test_power_prox_outside_fp32_range():
    """Magnitudes the FP32 start refuses take the FP64 iteration; a NaN stays a NaN."""
    import torch
    L = lib()
    p = dict(mi.small(seed=8, dim=2, nx=4, ny=6, nt=3, bc=("periodic", "periodic"))["problem"], qprime=3.0)
    zero = np.zeros(p["n"])
    rng = np.random.Generator(np.random.PCG64(3))
    for scale in (1e-14, 1e13):
        v = scale * rng.uniform(0.1, 1.0, size=(5, p["nt"]) + tuple(p["n"]))
        y = torch.empty(v.size, dtype=torch.float64, device="cuda")
        L.mfg_prox(L.mfg_plan(p), 0, 0.7, dev(v), dev(zero), dev(zero), y)
        ref = oracle_prox(p, 0.7, v, zero, zero).reshape(-1)
        assert np.abs(host(y) - ref).max() <= 1e-12 * np.abs(ref).max()
    v[0, 1, 2, 3] = np.nan
    L.mfg_prox(L.mfg_plan(p), 0, 0.7, dev(v), dev(zero), dev(zero), y)
    out = host(y).reshape(v.shape)
    assert np.isnan(out[:, 1, 2, 3]).all() and np.isfinite(out[0]).sum() == out[0].size - 1
