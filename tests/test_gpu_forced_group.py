"""A forced number of frequencies per pass, spread evenly over its passes, is what runs, with the
cluster size left to the library or not, in formal solutions and in emergent profiles' sweep (the
same rule); only where no cluster size holds it do the frequencies go into smaller passes.
"""
import pytest

import paper_1307_4217_gb300 as P
from gpu_util import initial_rho, make_ctx, polarized_case, unpolarized_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [P.PORTA_FP32, P.PORTA_FP64])
@pytest.mark.parametrize("model", [0, 1])
@pytest.mark.parametrize("n,n_nu", [(8, 7), (16, 21), (5, 9), (24, 11)])
def test_group_is_kept(n, n_nu, model, prec):
    atm = polarized_case(n, n, 6, seed=3) if model else unpolarized_case(n, n, 6, seed=3)
    rho = initial_rho(atm, model)
    for f in {1, 2, 3, 4, n_nu // 2, n_nu}:
        passes = -(-n_nu // f)
        even = -(-n_nu // passes)
        ctx = make_ctx(atm, model, 2, 4, n_nu, prec, rho=rho, nu_group=f)
        ctx.formal_solve()
        assert ctx.launch_info()["nu_group"] == even, f
        ctx.close()


def test_group_that_fits_nowhere_is_split():
    atm = polarized_case(64, 64, 4, seed=3)
    # (12 frequencies of 64 columns fit the general sweep, as a forced shape must, not this one)
    ctx = make_ctx(atm, 1, 1, 2, 12, P.PORTA_FP32, rho=initial_rho(atm, 1), nu_group=12)
    ctx.formal_solve()
    assert 1 <= ctx.launch_info()["nu_group"] < 12
