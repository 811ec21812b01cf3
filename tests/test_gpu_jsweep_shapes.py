"""The J^K_Q sweep kernels at the edges of their tiling, against the FP64 oracle: odd and
single frequencies (a half-empty lane pair), two and three planes (no halo row overwritten),
strips of one row, strips of unequal height, points in several rounds of a CTA's threads,
several groups of threads per point, and planes too wide for the four-slot kernel.

Tolerances: those of the parity tests. FP32 1e-5 (J^0_0 and Lambda-bar* relative, the
other components relative to J^0_0): an FP32 step rounds a few times 2^-24 and the sums over
rays and frequencies average, so 1e-5 leaves a factor of about 50. FP64 1e-10.
"""
import numpy as np
import pytest

import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, oracle_fs, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu

F32, F64 = P.PORTA_FP32, P.PORTA_FP64
# nx, ny, nz, n_nu, cluster, nu_group (0: automatic)
SHAPES = [
    (5, 3, 2, 1, 1, 0), (5, 3, 3, 2, 3, 1), (7, 5, 4, 3, 2, 3), (7, 5, 9, 5, 5, 2), (9, 16, 6, 4, 16, 0),
    (33, 9, 5, 7, 4, 0), (48, 13, 4, 5, 1, 2), (31, 17, 5, 6, 7, 4), (16, 11, 6, 9, 3, 0),
]


def _check(jg, lg, jo, lo, tol):
    s = np.abs(jo[..., :1])
    assert np.max(np.abs(jg - jo) / s) < tol
    assert np.max(np.abs(lg - lo) / np.abs(lo)) < tol


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("prec", [F32, F64])
@pytest.mark.parametrize("nx,ny,nz,n_nu,cluster,nu_group", SHAPES)
def test_shape(nx, ny, nz, n_nu, cluster, nu_group, prec, model):
    atm = polarized_case(nx, ny, nz, seed=nx + nz) if model else unpolarized_case(nx, ny, nz, seed=nx)
    rho = initial_rho(atm, model, seed=ny)
    if prec == F64 and (nx, cluster) == (48, 1):
        cluster = 2                     # (one strip of 48 x 13 points does not fit in FP64)
    ctx = make_ctx(atm, model, 2, 4, n_nu, prec, rho=rho, cluster=cluster, nu_group=nu_group)
    ctx.formal_solve()
    jg, lg = ctx.accumulate_jkq()
    _, (jo, lo) = oracle_fs(atm, model, 2, 4, n_nu, rho)
    _check(jg, lg, jo, lo, 1e-5 if prec == F32 else 1e-10)


@pytest.mark.parametrize("nx,ny,prec", [(200, 60, F32), (104, 52, F64)])
def test_wide_plane(nx, ny, prec):
    atm = polarized_case(nx, ny, 4, seed=5)
    rho = initial_rho(atm, 1, seed=6)
    ctx = make_ctx(atm, 1, 2, 4, 3, prec, rho=rho)
    ctx.formal_solve()
    jg, lg = ctx.accumulate_jkq()
    _, (jo, lo) = oracle_fs(atm, 1, 2, 4, 3, rho)
    _check(jg, lg, jo, lo, 1e-5 if prec == F32 else 1e-10)


@pytest.mark.parametrize("prec", [F32, F64])
def test_no_room_for_packed_inputs(prec):
    """The sums fit the device limit, the packed inputs do not: another kernel takes over."""
    atm = polarized_case(12, 10, 8, seed=3)
    rho = initial_rho(atm, 1, seed=4)
    ctx = make_ctx(atm, 1, 2, 4, 5, prec, rho=rho)
    nvox = 12 * 10 * 8
    sums = nvox * (7 * 8 + 4) if prec == F32 else nvox * 16 * 4 * 8      # rays x 4 partials in FP64
    assert P.porta_set_device_limit(P.porta_device_bytes() + sums + 4096) == P.PORTA_OK
    try:
        ctx.formal_solve()
        jg, lg = ctx.accumulate_jkq()
    finally:
        assert P.porta_set_device_limit(0) == P.PORTA_OK
    _, (jo, lo) = oracle_fs(atm, 1, 2, 4, 5, rho)
    _check(jg, lg, jo, lo, 1e-5 if prec == F32 else 1e-10)
