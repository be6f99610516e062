"""The mixed-radix FFT passes over every radix, their compositions, odd and even
lengths, both axes, the smallest and largest lengths, blocks with a partial last
pair of lines, and both boundary conditions, against the assembled P by normwise
backward error (the bars of the other preconditioner tests, 1e-12 and 5e-5)."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle import operators as ops

from _gpu_helpers import dev, host, lib

pytestmark = pytest.mark.gpu

LENGTHS = [9, 10, 11, 12, 13, 14, 20, 24, 30, 49, 60, 75, 99, 104, 121, 150, 169, 200, 243, 360, 500]


def _check(p, precision, bar):
    import torch
    L = lib()
    n = ops.sizes(p)[1]
    plan = L.mfg_plan(p, precision=precision)
    assert L.mfg_get_schedule(plan, 0)["fft"][0] == 1
    r = mi.random_field(n, 9)
    z = torch.empty(n, dtype=torch.float64, device="cuda")
    L.mfg_apply_precond(plan, 0, dev(r), z)
    P, zh = ops.precond(p), host(z)
    eta = np.abs(r - P @ zh).max() / (abs(P).sum(axis=1).max() * np.abs(zh).max() + np.abs(r).max())
    assert eta <= bar


@pytest.mark.parametrize("n", LENGTHS + [1024, 1500, 2048])
@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-12), ("mixed", 5e-5)])
def test_lines_along_y(n, bc, precision, bar):
    _check(mi.small(seed=n, dim=1, nx=n, nt=3, bc=(bc, "periodic"), nu=0.05)["problem"], precision, bar)


@pytest.mark.parametrize("n", LENGTHS[::2])
@pytest.mark.parametrize("bc", ["periodic", "neumann"])
@pytest.mark.parametrize("precision,bar", [("fp64", 1e-12), ("mixed", 5e-5)])
def test_lines_along_x(n, bc, precision, bar):
    _check(mi.small(seed=n, dim=2, nx=n, ny=19, nt=2, bc=(bc, "neumann"), nu=0.05)["problem"], precision, bar)
