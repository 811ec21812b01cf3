"""The emergent sweep with its shape forced, at the edges of its tiling: half-empty frequency
pairs, two and three planes, strips of one row and of unequal height, several passes, several
rounds and groups of threads. The profiles against the FP64 oracle's, and the reverse mode's
gradients, which read the Stokes vectors that the sweep stores of every node, against those of
the oracle from FP64 stores.

Tolerances: those of the parity tests of the same calls. FP32 profiles 1e-5 of the largest
intensity; FP64 1e-10 for profiles and gradients, the latter relative to their largest element.
"""
import numpy as np
import pytest

import oracle
import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu

F32, F64 = P.PORTA_FP32, P.PORTA_FP64
# nx, ny, nz, n_nu, cluster, nu_group
SHAPES = [(5, 3, 2, 1, 1, 1), (5, 3, 3, 2, 3, 1), (7, 5, 4, 3, 2, 3), (7, 5, 9, 5, 5, 2), (9, 16, 6, 4, 16, 4),
          (33, 9, 5, 7, 4, 7), (31, 17, 5, 6, 7, 4), (16, 11, 6, 9, 3, 5), (48, 13, 4, 5, 1, 2), (40, 24, 4, 3, 3, 1)]
MU, CHI = np.array([1.0, 0.35, 0.6]), np.array([0.0, 0.7, 4.2])


def _case(nx, ny, nz, n_nu, cluster, nu_group, prec, model):
    atm = polarized_case(nx, ny, nz, seed=nx + nz) if model else unpolarized_case(nx, ny, nz, seed=nx)
    rho = initial_rho(atm, model, seed=ny)
    # (a varying source function: control points away from the kink at equal ones)
    rho[..., 0] *= np.exp(0.2 * np.random.default_rng(ny).normal(size=rho.shape[:-1]))
    if prec == F64 and (nx, cluster) == (48, 1):
        cluster = 2                     # (one strip of 48 x 13 points does not fit in FP64)
    ctx = make_ctx(atm, model, 2, 4, n_nu, prec, rho=rho, cluster=cluster, nu_group=nu_group)
    return ctx, oracle.Problem(atm, model, 2, 4, n_nu), rho


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("prec", [F32, F64])
@pytest.mark.parametrize("shape", SHAPES)
def test_profiles(shape, prec, model):
    ctx, prob, rho = _case(*shape, prec, model)
    out = np.asarray(ctx.emergent_stokes(MU, CHI))
    ref = np.asarray(oracle.emergent(prob, rho, MU, CHI)).reshape(out.shape)
    assert np.max(np.abs(out - ref)) < (1e-5 if prec == F32 else 1e-10) * np.max(np.abs(ref))


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("shape", SHAPES)
def test_gradients(shape, model):
    ctx, prob, rho = _case(*shape, F64, model)
    g = np.random.default_rng(3).normal(size=(len(MU), shape[3], shape[1], shape[0], 4 if model else 1))
    got = ctx.emergent_vjp(MU, CHI, g)
    want = oracle.emergent_vjp(prob, rho, MU, CHI, g)
    for a, b in list(zip(got, want))[: 3 if model else 2]:
        assert np.max(np.abs(np.asarray(a).reshape(b.shape) - b)) < 1e-10 * np.max(np.abs(b))
