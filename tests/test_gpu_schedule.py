"""mfg_get_schedule reports the blocks of the AAt launch: column blocks (32 x 8 columns,
chunks of planes) for a viscosity field and the double-float stencil, warp strips
otherwise, by the default launch rules written out here."""
import math

import numpy as np
import pytest

import mfg_inputs as mi

from _gpu_helpers import lib

pytestmark = pytest.mark.gpu

WANT = 152 * 8


def _columns(nx, ny, nt):
    cols = math.ceil(ny / 32) * math.ceil(nx / 8)
    kc = math.ceil(nt / min(nt, math.ceil(WANT / cols)))
    return cols * math.ceil(nt / kc)


def _strips(nx, ny, nt, per_sm):
    """Least waves x (rows + 1.5), chunks of 2 to 32 rows; blocks of 8 warps, fewer
    where that leaves fewer than 4 blocks per SM."""
    base, best = math.ceil(ny / 32) * nt, None
    for want in range(32, 1, -1):
        rows = math.ceil(nx / math.ceil(nx / want))
        blocks = math.ceil(base * math.ceil(nx / want) / 8)
        cost = math.ceil(blocks / (WANT // 8 * per_sm)) * (rows + 1.5)
        if best is None or cost < best[0]:
            best = (cost, rows)
    items, warps = base * math.ceil(nx / best[1]), 8
    while warps > 1 and items < warps * 152 * 4:
        warps //= 2
    return math.ceil(items / warps)


@pytest.mark.parametrize("nx,ny,nt", [(1, 64, 32), (40, 40, 16), (201, 147, 50), (512, 512, 16)])
def test_aat_blocks(nx, ny, nt):
    L = lib()
    dim = 1 if nx == 1 else 2
    n = (ny, 1) if dim == 1 else (nx, ny)
    p = mi.small(seed=1, dim=dim, nx=n[0], ny=n[1], nt=nt, bc=("neumann", "periodic"))["problem"]
    blocks = lambda q, precision: L.mfg_get_schedule(L.mfg_plan(q, precision=precision), 0)["aat_blocks"]
    assert blocks(p, "mixed") == max(_strips(nx, ny, nt, 4), _strips(nx, ny, nt, 3))
    assert blocks(p, "mixed_df") == _columns(nx, ny, nt)
    if nx * ny <= 1600:
        assert blocks(dict(p, nu_field=np.full(n, 0.1)), "mixed") == _columns(nx, ny, nt)


def test_square_and_oblong_cells_are_tuned_apart():
    """They run different stencil kernels, so a choice timed for one is not taken for the other."""
    L = lib()
    p = mi.small(seed=1, dim=2, nx=44, ny=44, nt=6, bc=("periodic", "periodic"))["problem"]
    measured = []
    for length in ((1.0, 1.0), (1.0, 2.0), (2.0, 2.0), (1.0, 3.0)):
        plan = L.mfg_plan(dict(p, len=length), precision="mixed")
        L.mfg_autotune(plan)
        measured.append(L.mfg_get_schedule(plan, 0)["measured"])
    assert measured == [1, 1, 0, 0]
