"""The active set of the adjoint is read off y (m > 0, w != 0), also where w/m
underflows: fluxes of the smallest subnormal number against the oracle's sparse KKT
solve.  Bar of the existing adjoint tests (1e-7)."""
import numpy as np
import pytest

import mfg_inputs as mi
from oracle import adjoint as oadj

from _gpu_helpers import dev, host, lib, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [10, 32])
def test_tiny_fluxes_are_active(ny):
    import torch
    p = mi.small(seed=4, dim=2, nx=6, ny=ny, nt=4, bc=("neumann", "periodic"), nu=0.1)["problem"]
    shp = (5, 4, 6, ny)
    rng = np.random.Generator(np.random.PCG64(5))
    y = rng.uniform(3.0, 5.0, size=shp)
    y[2::2] *= -1.0
    y[1:, :, ::2, ::3] = np.array(5e-324) * np.array([1, -1, 1, -1]).reshape(4, 1, 1, 1)
    z, g = np.zeros(shp[1:]), rng.normal(size=shp)
    ref = oadj.adjoint_gradients(p, y, z, g)
    out = {k: torch.empty(6 * ny, dtype=torch.float64, device="cuda") for k in ("dm0", "dV", "dW")}
    dnu = torch.empty(1, dtype=torch.float64, device="cuda")
    rc, _ = lib().mfg_adjoint(lib().mfg_plan(p), 0, dev(y), dev(z), dev(g), out["dm0"], out["dV"], out["dW"], dnu, tol=1e-12)
    assert rc == 0
    for k in out:
        assert rel(host(out[k]), ref[k]) <= 1e-7
