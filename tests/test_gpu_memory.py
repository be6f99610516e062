"""What a plan can do without is not taken from memory that is short: with the
device filled up, plans are built and calls answered as in the memory their
mandatory workspace takes.  Both sides evaluate the same formulas, so the bars are
those of the tests against the oracle (1e-12 for P^{-1} in FP64, 1e-7 for gradients)."""
import numpy as np
import pytest

import mfg_inputs as mi

from _gpu_helpers import lib

pytestmark = pytest.mark.gpu


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _fill(leave):
    import torch
    return torch.empty(max(0, _free() - int(leave)), dtype=torch.uint8, device="cuda")


def _rel(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("l", [1, 2])
def test_plan_without_room_for_the_time_factors(l):
    import torch
    L = lib()
    p = mi.small(seed=1, dim=2, nx=256, ny=256, nt=256, bc=("periodic", "neumann"), l=l)["problem"]
    n = 256 ** 3
    r = torch.randn(n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    ref, z = torch.empty_like(r), torch.empty_like(r)
    for _ in range(2):  # the first pass loads the kernels
        before = _free()
        plan = L.mfg_plan(p, precision="fp64")
        used = before - _free()
        L.mfg_apply_precond(plan, 0, r, ref)
        torch.cuda.synchronize()
        L.mfg_destroy(plan)
    fill = _fill(used - 4 * n)  # the factors are 8 n bytes
    plan = L.mfg_plan(p, precision="fp64")
    L.mfg_apply_precond(plan, 0, r, z)
    torch.cuda.synchronize()
    L.mfg_destroy(plan)
    del fill
    assert _rel(z, ref) <= 1e-12
