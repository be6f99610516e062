"""The AAt apply over the shapes of its launch: strips of 32 columns with every
kind of last strip, row chunks of one to 32 rows and several chunks, the
shortest axes and time grids, square cells (shared pair sums) and oblong ones,
each boundary condition, against the oracle's sparse matrix at the operators'
bar (1e-12, relative l2 and l_inf)."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle import operators as ops

from _gpu_helpers import dev, host, lib, linf_rel, rel

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 2), (3, 31, 2), (33, 32, 3), (8, 33, 2), (65, 63, 2), (70, 64, 5), (9, 97, 40), (40, 2, 7), (128, 128, 3)]


@pytest.mark.parametrize("nx,ny,nt", SHAPES)
@pytest.mark.parametrize("bc", [("periodic", "neumann"), ("neumann", "periodic"), ("neumann", "neumann"),
                                ("periodic", "periodic")])
@pytest.mark.parametrize("square", [True, False])
def test_aat_shapes(nx, ny, nt, bc, square):
    import torch
    p = mi.small(seed=nx + ny, dim=2, nx=nx, ny=ny, nt=nt, bc=bc, nu=0.3)["problem"]
    if square:  # equal spacings, exactly: lengths that are the (power-of-two scaled) cell counts
        cells = [n if b == "periodic" else n + 1 for n, b in zip((nx, ny), bc)]
        p["len"] = (cells[0] / 64.0, cells[1] / 64.0)
    L = lib()
    n = ops.sizes(p)[1]
    v = mi.random_field(n, 3)
    q = torch.empty(n, dtype=torch.float64, device="cuda")
    L.mfg_apply_AAt(L.mfg_plan(p), 0, dev(v), q)
    ref = ops.AAt(p) @ v
    assert rel(host(q), ref) <= 1e-12 and linf_rel(host(q), ref) <= 1e-12
