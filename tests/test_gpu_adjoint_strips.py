"""The adjoint over the shapes its operators run in: strips and point by point, several
strips, ragged last strips, several row chunks, both boundary conditions, against the
oracle's sparse KKT solve.  Bar of the existing adjoint tests (1e-7)."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle import adjoint as oadj

from _gpu_helpers import dev, host, lib, rel

pytestmark = pytest.mark.gpu

CASES = [  # nx, ny, bc: H^-1 C^T and (2-D) C in strips from 7/8 of the lanes on
    (5, 21, ("periodic", "neumann")),
    (9, 45, ("neumann", "periodic")),
    (12, 70, ("periodic", "neumann")),
    (40, 28, ("periodic", "periodic")),  # at the line
    (6, 60, ("neumann", "neumann")),     # two strips, the last ragged
    (70, 1, ("neumann", "periodic")),    # 1-D
]


@pytest.mark.parametrize("nx,ny,bc", CASES)
def test_adjoint_of_ragged_strips(nx, ny, bc):
    import torch
    dim = 1 if ny == 1 else 2
    p = mi.small(seed=6, dim=dim, nx=nx, ny=ny, nt=3, bc=bc, nu=0.1)["problem"]
    shp = (1 + 2 * dim, 3, nx, ny)
    rng = np.random.Generator(np.random.PCG64(7))
    y = rng.uniform(1.0, 2.0, size=shp)
    y[2::2] *= -1.0
    y[1:] *= rng.uniform(size=y[1:].shape) < 0.6
    y[0, 1, ::3] = 0.0
    z, g = rng.normal(size=shp[1:]), rng.normal(size=shp)
    ref = oadj.adjoint_gradients(p, y, z, g)
    out = {k: torch.empty(nx * ny, dtype=torch.float64, device="cuda") for k in ("dm0", "dV", "dW")}
    dnu = torch.empty(1, dtype=torch.float64, device="cuda")
    rc, _ = lib().mfg_adjoint(lib().mfg_plan(p), 0, dev(y), dev(z), dev(g), out["dm0"], out["dV"], out["dW"], dnu, tol=1e-12)
    assert rc == 0
    for k in out:
        assert rel(host(out[k]), ref[k]) <= 1e-7
    assert abs(host(dnu)[0] - ref["dnu"]) <= 1e-7 * max(1.0, abs(ref["dnu"]))
