"""No bias of the FP32 sums: over a thick polarized box the mean relative errors against FP64 of
J^0_0 in every plane, and of Lambda-bar* in the planes where it exceeds 0.9 and the update divides
by what is left of 1, stay below 1e-8. A plane has 24 x 20 voxels whose errors (4e-8 rms: a few
FP32 roundings averaged over 48 to 160 rays) are independent, so that their mean is 2e-9 and 1e-8
leaves a factor of 5. What would not average out: the rounding of the profile's norm and of the
ray weights, the same for all voxels (1e-8 to 3e-8), and that of the reciprocal in kappa^-1,
one-sided (2.5e-8 of the intensity).
"""
import numpy as np
import pytest

import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, polarized_case

pytestmark = pytest.mark.gpu
QUADS = [(5, 16, 21), (4, 10, 21), (3, 8, 11)]


def _errors(quad):
    atm = polarized_case(24, 20, 16, seed=3)
    atm["chi"] = atm["chi"] * 30.0
    rho = initial_rho(atm, 1, seed=4)
    out = []
    for prec in (P.PORTA_FP32, P.PORTA_FP64):
        ctx = make_ctx(atm, 1, *quad, prec, rho=rho)
        ctx.formal_solve()
        j, l = ctx.accumulate_jkq()
        out.append((np.asarray(j)[..., 0].reshape(16, -1), np.asarray(l).reshape(16, -1)))
    (j32, l32), (j64, l64) = out
    return ((j32 - j64) / j64).mean(1), ((l32 - l64) / l64).mean(1), l64.mean(1)


@pytest.mark.parametrize("quad", QUADS)
def test_lambda_of_thick_planes(quad):
    _, err, lam = _errors(quad)
    assert np.sum(lam > 0.9) >= 4
    assert np.max(np.abs(err[lam > 0.9])) < 1e-8


@pytest.mark.parametrize("quad", QUADS)
def test_mean_intensity(quad):
    err, _, _ = _errors(quad)
    assert np.max(np.abs(err)) < 1e-8
