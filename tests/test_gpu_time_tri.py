"""The time pass as a tridiagonal elimination per spatial mode, over the block
shapes it launches (32, 64 and 128 threads, partial last blocks, the longest
time axis, which fills a warp's shared memory) and over coefficients from nearly
singular modes (long horizon, no viscosity) to dominant ones, against the
assembled P by normwise backward error.

Bars: the elimination adds a few roundings per element to the transforms', so
the bars of the other preconditioner tests hold, 1e-12 in FP64 and 5e-5 in FP32."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle import operators as ops

from _gpu_helpers import dev, host, lib

pytestmark = pytest.mark.gpu

CASES = [
    dict(seed=1, dim=1, nx=33, nt=2, bc=("neumann", "periodic")),
    dict(seed=2, dim=1, nx=31, nt=256, bc=("periodic", "periodic")),
    dict(seed=3, dim=2, nx=9, ny=13, nt=255, bc=("neumann", "periodic"), nu=0.0),
    dict(seed=4, dim=2, nx=67, ny=75, nt=5, bc=("periodic", "neumann")),            # 64-thread blocks
    dict(seed=5, dim=2, nx=160, ny=128, nt=3, bc=("neumann", "neumann"), nu=1.0),   # 128-thread blocks
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("l", [1, 2])
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-12), ("mixed", 5e-5)])
def test_time_elimination(case, l, precision, bar):
    import torch
    p = mi.small(**dict(case, l=l))["problem"]
    L = lib()
    n = ops.sizes(p)[1]
    P = ops.precond(p)
    r = mi.random_field(n, 5)
    r[::3] = 1.0  # a share of the constant mode, the nearly singular one
    z = torch.empty(n, dtype=torch.float64, device="cuda")
    L.mfg_apply_precond(L.mfg_plan(p, precision=precision), 0, dev(r), z)
    zh = host(z)
    eta = np.abs(r - P @ zh).max() / (abs(P).sum(axis=1).max() * np.abs(zh).max() + np.abs(r).max())
    assert eta <= bar
