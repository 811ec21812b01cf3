"""Rays along a grid axis, whose component across it is 1e-17 and not 0: they stay on their line
of nodes. A nearly transparent box carries the bottom's Planck function, a different one under
every column, to the top through 64 planes; along an axis only the neighbours on the ray's line
may mix. FP32 against the FP64 oracle: a plane rounds an intensity about twice, 2^-25 rms each,
so 64 planes leave 3.4e-7 rms, and 1e-6 leaves a factor of 3. (A leak of one rounding unit of
the weight per plane, 2^-24, gives 64 x 6e-8 times the contrast, above 3e-6.)
"""
import numpy as np
import pytest

import oracle
import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu


def _box(model):
    atm = polarized_case(16, 12, 64, seed=3) if model else unpolarized_case(16, 12, 64, seed=3)
    atm["chi"] = np.full_like(atm["chi"], 1e-9)
    rng = np.random.default_rng(7)
    atm["bpl"][0] = np.exp(rng.normal(size=atm["bpl"][0].shape))
    return atm, initial_rho(atm, model)


def _rms(a, b):
    return float(np.sqrt(np.mean((a - b) ** 2) / np.mean(b**2)))


@pytest.mark.parametrize("model", [0, 1])
def test_emergent_profiles(model):
    atm, rho = _box(model)
    ctx = make_ctx(atm, model, 1, 2, 4, P.PORTA_FP32, rho=rho)
    mu, chi = np.full(4, 0.5), np.arange(4) * 0.5 * np.pi
    out = np.asarray(ctx.emergent_stokes(mu, chi))
    ref = oracle.emergent(oracle.Problem(atm, model, 1, 2, 4), rho, mu, chi).reshape(out.shape)
    for d in range(4):
        assert _rms(out[d][..., 0], ref[d][..., 0]) < 1e-6, d


@pytest.mark.parametrize("model", [0, 1])
def test_mean_intensity(model):
    # azimuths pi / 2 and 3 pi / 2
    atm, rho = _box(model)
    ctx = make_ctx(atm, model, 2, 2, 4, P.PORTA_FP32, rho=rho)
    ctx.formal_solve()
    j, _ = ctx.accumulate_jkq()
    jo, _ = oracle.formal_solve(oracle.Problem(atm, model, 2, 2, 4), rho)
    j, jo = np.asarray(j), np.asarray(jo).reshape(np.asarray(j).shape)
    assert _rms(j[-1, ..., 0], jo[-1, ..., 0]) < 1e-6
