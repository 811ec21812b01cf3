"""The rounding of a node's weight w_m / (chi N) does not go into J^0_0 undiminished. In a
transparent box over a uniform bottom every voxel of a plane has the same J^0_0, and its opacity
and velocity, different ones everywhere, enter only through FP32 roundings. Those of the
profiles, products and sums differ from ray to ray and average out over the 32 upward rays; that
of the weight, 2^-25 to 2^-24 at most or 2.5e-8 rms, is the same for all rays of one w_m when it is
rounded to the nearest. The rest alone is 2.4e-8 (2.2e-8 polarized), as it is for weights that are
not divided by chi; with the weight to the nearest it is the root of the sum of the squares, 3.5e-8
(3.3e-8). The bound of 3e-8 lies between.
"""
import numpy as np
import pytest

import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [0, 1])
def test_spread_over_a_plane(model):
    atm = polarized_case(32, 32, 6, seed=3) if model else unpolarized_case(32, 32, 6, seed=3)
    rng = np.random.default_rng(5)
    atm["chi"] = 1e-16 * np.exp(rng.normal(size=atm["chi"].shape))
    atm["bpl"] = np.ones_like(atm["bpl"])
    ctx = make_ctx(atm, model, 4, 8, 61, P.PORTA_FP32, rho=initial_rho(atm, model))
    ctx.formal_solve()
    j, _ = ctx.accumulate_jkq()
    j = np.asarray(j)[..., 0].reshape(6, -1)
    assert np.sqrt(np.mean((np.std(j, axis=1) / np.mean(j, axis=1)) ** 2)) < 3e-8
