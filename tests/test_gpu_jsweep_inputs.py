"""The J^K_Q sweep without room for its packed inputs: it copies the same values from where
they are, so J^K_Q, Lambda-bar*, iterations, emergent profiles and gradients are those with
them to the last bit, whatever launch shape or filler was set before the room ran out, and the
packed inputs come back with new unknowns once there is room.
"""
import numpy as np
import pytest
import torch

import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu

F32, F64 = P.PORTA_FP32, P.PORTA_FP64
NX, NY, NZ, NNU = 12, 10, 8, 5
MU, CHI = [1.0, 0.4], [0.0, 1.1]


def _ctx(model, prec, **kw):
    atm = polarized_case(NX, NY, NZ, seed=3) if model else unpolarized_case(NX, NY, NZ, seed=3)
    rho = initial_rho(atm, model, seed=4)
    return make_ctx(atm, model, 2, 4, NNU, prec, rho=rho, **kw), rho


def _sums_bytes(model, prec):
    nvox = NX * NY * NZ
    if prec == F32:
        return nvox * ((7 if model else 2) * 8 + 4)
    return nvox * 16 * (4 if model else 2) * 8      # rays x partials


def _no_room(n):
    assert P.porta_set_device_limit(P.porta_device_bytes() + n) == P.PORTA_OK


def _run(ctx):
    ctx.formal_solve()
    j, l = ctx.accumulate_jkq()
    return np.asarray(j), np.asarray(l)


@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("prec", [F32, F64])
def test_same_sums_and_room_again(prec, model):
    full, rho = _ctx(model, prec)
    jf, lf = _run(full)
    ctx, rho = _ctx(model, prec)
    words = (12 if model else 4) * NX * NY * NZ * (4 if prec == F32 else 8)
    _no_room(_sums_bytes(model, prec) + words // 2)
    try:
        before = P.porta_device_bytes()
        j, l = _run(ctx)
        assert P.porta_device_bytes() - before < _sums_bytes(model, prec) + words // 2
    finally:
        assert P.porta_set_device_limit(0) == P.PORTA_OK
    assert np.array_equal(j, jf) and np.array_equal(l, lf)
    before = P.porta_device_bytes()
    ctx.set_rho(rho)
    j, l = _run(ctx)
    assert P.porta_device_bytes() - before == words
    assert np.array_equal(j, jf) and np.array_equal(l, lf)


@pytest.mark.parametrize("prec", [F32, F64])
def test_filler_set_before_the_room_ran_out(prec):
    full, _ = _ctx(1, prec)
    ctx, _ = _ctx(1, prec)
    for c in (full, ctx):
        c.set_fill(2, 1, 0.3)
    jf, lf = _run(full)
    _no_room(_sums_bytes(1, prec) + 4096)
    try:
        j, l = _run(ctx)
    finally:
        assert P.porta_set_device_limit(0) == P.PORTA_OK
    assert ctx.fill_info() == full.fill_info()
    assert np.array_equal(j, jf) and np.array_equal(l, lf)


def test_iterations_by_graph():
    full, _ = _ctx(1, F32)
    ctx, _ = _ctx(1, F32)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for c, s in zip((full, ctx), streams):
        c.set_stream(s.cuda_stream)
    rf = full.run_iterations(3)
    _no_room(_sums_bytes(1, F32) + 4096)
    try:
        r = ctx.run_iterations(2)
    finally:
        assert P.porta_set_device_limit(0) == P.PORTA_OK
    r = ctx.run_iterations(1)
    assert r == rf
    assert np.array_equal(ctx.get_rho(), full.get_rho())


@pytest.mark.parametrize("prec", [F32, F64])
def test_emergent_profiles(prec):
    full, _ = _ctx(1, prec)
    ref = np.asarray(full.emergent_stokes(MU, CHI))
    ctx, _ = _ctx(1, prec)
    nout = 2 * NNU * NX * NY * 4 * 8
    _no_room(nout + 16384)
    try:
        out = np.asarray(ctx.emergent_stokes(MU, CHI))
    finally:
        assert P.porta_set_device_limit(0) == P.PORTA_OK
    assert np.array_equal(out, ref)


def test_wide_planes_take_their_own_kernel():
    """FP32 planes too wide for the four-slot kernel: fixed-point sums, but no packed inputs (nor
    the per-ray partials of the general sweep)."""
    atm = polarized_case(200, 60, 4, seed=5)
    ctx = make_ctx(atm, 1, 2, 4, 3, F32, rho=initial_rho(atm, 1, seed=6))
    before = P.porta_device_bytes()
    ctx.formal_solve()
    assert P.porta_device_bytes() - before == 200 * 60 * 4 * (7 * 8 + 4)
