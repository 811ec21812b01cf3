"""The unit of length does not matter: opacities times 2^-k over heights and periods times 2^k give
the same J^K_Q and Lambda-bar* in FP32, down to opacities of 2^-92 (2e-28) times the source
function. Every optical path is the same number; what differs is rounded at the lower end of the
FP32 range (products of opacity, profile, source function and weights that become subnormal),
a few 2^-24 at most: 1e-6 of J^0_0.
"""
import numpy as np
import pytest

import paper_1307_4217_gb300 as P
from gpu_util import polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu


def _solve(atm, model, k):
    a = dict(atm)
    a["chi"], a["z"] = atm["chi"] * 2.0**-k, atm["z"] * 2.0**k
    a["lx"], a["ly"] = atm["lx"] * 2.0**k, atm["ly"] * 2.0**k
    rho = np.zeros(a["chi"].shape + (6 if model else 1,))
    rho[..., 0] = a["bpl"]
    ctx = P.Context(a, model, 2, 4, 5, 1.5, precision=P.PORTA_FP32)
    ctx.set_atmosphere(a)
    ctx.set_rho(rho)
    ctx.formal_solve()
    j, l = ctx.accumulate_jkq()
    return np.asarray(j), np.asarray(l)


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("k", [40, 70, 85, -40, -70])
def test_unit_of_length(k, model):
    atm = polarized_case(8, 8, 6, seed=3) if model else unpolarized_case(8, 8, 6, seed=3)
    rng = np.random.default_rng(3)
    atm["chi"] = np.exp(0.5 * rng.normal(size=atm["chi"].shape)) / 128.0
    atm["z"] = np.arange(6) * 100.0
    atm["lx"] = atm["ly"] = 800.0
    atm["vel"] = 0.1 * rng.normal(size=atm["chi"].shape)
    j0, l0 = _solve(atm, model, 0)
    j, l = _solve(atm, model, k)
    assert np.max(np.abs(j - j0) / np.abs(j0[..., :1])) < 1e-6
    assert np.max(np.abs(l - l0)) < 1e-6
