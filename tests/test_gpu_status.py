"""Errors that a formal solution finds out on the device are reported by the next call that
synchronizes for a residual, the unknowns or J^K_Q, also where a later formal solution of the
same call was clean; each once. The first iteration overflows the fixed-point range (a voxel
2^30 times as bright as its neighbours' source and Planck functions, beyond the 2^16 of headroom
even after the smallest ray weight, 1/64); the voxel itself emits little (its optical path is
short), so that the iterations after it are clean.
"""
import numpy as np
import pytest
import torch

import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu


def _raises(what):
    with pytest.raises(P.PortaError) as e:
        what()
    assert e.value.code == P.PORTA_EKERNEL


def _ctx(model, n=8, nz=9, bright=True):
    atm = polarized_case(n, n, nz, seed=3) if model else unpolarized_case(n, n, nz, seed=3)
    ctx = P.Context(atm, model, 2, 4, 5, precision=P.PORTA_FP32)
    ctx.set_atmosphere(atm)
    good = initial_rho(atm, model)
    bad = good.copy()
    if bright:
        bad[nz - 2, 4, 4, 0] *= 2.0**30
    ctx.set_rho(bad)
    s = torch.cuda.Stream()
    ctx.set_stream(s.cuda_stream)
    ctx._keep = s
    return ctx, good


def _device_sums(ctx):
    j = torch.empty(ctx.nvox * ctx.nj, dtype=torch.float64, device="cuda")
    l = torch.empty(ctx.nvox, dtype=torch.float64, device="cuda")
    ctx.formal_solve()
    ctx.accumulate_jkq(j, l)


@pytest.mark.parametrize("model", [0, 1])
def test_iterations_by_graph(model):
    ctx, good = _ctx(model)
    _raises(lambda: ctx.run_iterations(8))
    ctx.set_rho(good)
    ctx.run_iterations(3)                       # (reported once)


def test_iterations_without_residual():
    ctx, _ = _ctx(1)
    ctx.run_iterations(8, residual=False)
    _raises(ctx.get_rho)
    ctx.get_rho()


def test_sums_on_the_device():
    ctx, good = _ctx(1)
    _device_sums(ctx)
    ctx.set_rho(good)
    ctx.formal_solve()
    _raises(ctx.accumulate_jkq)
    ctx.formal_solve()
    ctx.accumulate_jkq()


def test_update_with_residual():
    ctx, _ = _ctx(1)
    ctx.formal_solve()
    ctx.accumulate_jkq(want=False)
    _raises(ctx.see_update)


def test_checkpointed_iterations():
    ctx, _ = _ctx(1)
    _raises(lambda: ctx.iterate_ckpt(6, 2, residual=False))


def test_vcycle():
    ctx, _ = _ctx(1)
    ctx.mg_setup(2)
    _raises(lambda: ctx.mg_vcycle(4, 4, 4))


def test_solution_whose_sums_went_nowhere():
    ctx, good = _ctx(1)
    ctx.formal_solve()
    ctx.set_rho(good)
    ctx.formal_solve()
    ctx.accumulate_jkq()
    ctx.see_update()


def test_bounded_wait_runs_out():
    rc, seconds = P.porta_eval_halo_wait()
    assert rc == P.PORTA_EKERNEL
    assert 1.9 < seconds < 10.0            # the limit, and the tries before it is read
