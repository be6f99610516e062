"""The primal step on a NaN: every component of y and of ybar in the cells the NaN
reaches is NaN (fluxes that a warp skips because they are zero throughout, too),
and no other cell is touched."""
import numpy as np
import pytest

import mfg_inputs as mi

from _gpu_helpers import dev, host, lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["potential", "dual", "-dual"])
@pytest.mark.parametrize("ny", [20, 40])
def test_nan_reaches_all_components(where, ny):
    import torch
    p = mi.small(seed=3, dim=2, nx=5, ny=ny, nt=3, bc=("neumann", "neumann"))["problem"]
    shp = (3, 5, ny)
    y0 = np.zeros((5,) + shp)
    y0[0] = 1.0
    V, z = np.zeros(shp[1:]), np.zeros(shp)
    bad = np.zeros(shp, dtype=bool)
    if where == "potential":
        V[2, 9] = np.nan
        bad[:, 2, 9] = True
    else:
        z[1, 2, 9] = np.nan if where == "dual" else -np.nan
        for d in ((0, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (-1, 0, 0)):
            bad[1 + d[0], 2 + d[1], 9 + d[2]] = True
    y, ybar = dev(y0), torch.empty(y0.size, dtype=torch.float64, device="cuda")
    lib().mfg_prox_step(lib().mfg_plan(p), 0, 0.6, dev(z), y, ybar, dev(V), dev(np.zeros(shp[1:])))
    for out in (y, ybar):
        assert (np.isnan(host(out).reshape(y0.shape)) == bad[None]).all()
