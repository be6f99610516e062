"""What a plan can do without is not taken from memory that is short: with the
device filled up, plans are built and calls answered as in the memory their
mandatory workspace takes.  Both sides evaluate the same formulas, so the bars are
those of the tests against the oracle (1e-12 for P^{-1} in FP64, 1e-7 for gradients)."""
import contextlib

import pytest

import mfg_inputs as mi

from _gpu_helpers import lib

pytestmark = pytest.mark.gpu


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@contextlib.contextmanager
def _filled(leave):
    """The device filled up but for `leave` bytes."""
    import torch
    fill = torch.empty(max(0, _free() - int(leave)), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del fill
        torch.cuda.empty_cache()


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
    with _filled(used - 4 * n):  # the factors are 8 n bytes
        plan = L.mfg_plan(p, precision="fp64")
        L.mfg_apply_precond(plan, 0, r, z)
        torch.cuda.synchronize()
        L.mfg_destroy(plan)
    assert _rel(z, ref) <= 1e-12


def test_adjoint_without_room_for_the_cell_data():
    import torch
    L = lib()
    # nu keeps cond(AAt) u below 1e-8
    p = mi.small(seed=2, dim=2, nx=256, ny=256, nt=128, bc=("neumann", "periodic"), nu=1e-2)["problem"]
    n, c = 256 * 256 * 128, 5
    gen = torch.Generator("cuda").manual_seed(2)
    y = 0.5 + torch.rand((c, n), dtype=torch.float64, device="cuda", generator=gen)
    y[2::2] *= -1.0
    g = torch.randn((c, n), dtype=torch.float64, device="cuda", generator=gen)
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    outs = []
    for short in (False, True):
        plan = L.mfg_plan(p, precision="mixed")
        out = [torch.empty(256 * 256, dtype=torch.float64, device="cuda") for _ in range(3)]
        out.append(torch.empty(1, dtype=torch.float64, device="cuda"))
        # room for the two mandatory vectors (c n and n doubles) and half of the cell data
        with _filled((c + 1 + c / 2) * 8 * n) if short else contextlib.nullcontext():
            rc, st = L.mfg_adjoint(plan, 0, y.reshape(-1), z, g.reshape(-1), *out, tol=1e-12)
            torch.cuda.synchronize()
        L.mfg_destroy(plan)
        assert rc == 0 and st.status == 0
        outs.append(out)
    for a, b in zip(*outs):
        assert _rel(a, b) <= 1e-7
