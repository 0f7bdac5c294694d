"""GPU: scales whose precisions leave 2^+-1000, where the FP64 kernels divide, on every FP64 kernel form."""
import numpy as np
import pytest

import gabp_synth
from gpu_common import ensure_built, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [3e-303, 1e-150, 1e150, 1e303])
@pytest.mark.parametrize("opts", [dict(kernel=2), dict(kernel=1, tile_x=32, tile_y=8), dict(kernel=1, tile_x=128, tile_y=8)])
def test_fp64_kernels_out_of_the_fast_range(orc, gamma, opts):
    ensure_built()
    p = gabp_synth.make_problem(20, 18, 0.3, 2, n_uniform=60)
    fl = orc.build_factors(p.nx, p.ny, p.kappa, p.obs_x, p.obs_y, p.y, p.noise_var, gamma)
    with np.errstate(all="ignore"):
        mu_o, var_o, _ = orc.gabp(fl, 0.5, 12)
    with solver(p, "fp64", gamma=gamma, **opts) as s:
        s.iterate(12, 0.5)
        mu, var = s.marginals()
    ok = np.isfinite(mu_o) & np.isfinite(var_o)
    np.testing.assert_allclose(mu[ok], mu_o[ok], rtol=1e-10, atol=1e-10 * np.max(np.abs(mu_o[ok])))
    np.testing.assert_allclose(var[ok], var_o[ok], rtol=1e-10)
