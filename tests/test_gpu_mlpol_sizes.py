"""The rate equations of polarized atoms of every tile size of the refinement's inverse (M
unknowns beyond the populations: below, at and just above 32, 64 and 96, the largest), against
the FP64 elimination of the whole system.

Tolerance: 1e-11 of the largest unknown. The refinement ends when its correction is below
1e-13 of the solution, the elimination's backward error is a few 2^-53 times M.
"""
import numpy as np
import pytest

import paper_1307_4217_gb300 as P
import synth
from oracle import mlpol

pytestmark = pytest.mark.gpu

ATOMS = {             # levels J, lines (upper, lower); M = sum of (2J+1)^2 - 1
    8: ([0, 1], [(1, 0)]),
    32: ([1, 2], [(1, 0)]),
    40: ([0, 1, 1, 2], [(1, 0), (3, 1), (3, 2)]),
    64: ([0, 1, 2, 1, 2], [(3, 0), (3, 1), (4, 1), (4, 2)]),
    72: ([2, 3], [(1, 0)]),
    96: ([3, 3], [(1, 0)]),
    120: ([2, 3, 3], [(1, 0), (2, 0)]),
}


@pytest.mark.parametrize("m", sorted(ATOMS))
def test_refined_solve_of_every_size(m):
    J, lines = ATOMS[m]
    n = len(lines)
    atom = dict(J=np.array(J, float), E=np.linspace(0.0, 2.5, len(J)), lines=np.array(lines),
                A=np.geomspace(1e7, 6e7, n), eps=np.full(n, 1e-2))
    assert sum((2 * j + 1) ** 2 - 1 for j in J) == m
    atm = synth.multilevel_box(4, 3, 5, seed=m, tau_top=1e-3, tau_bot=1e2)
    atm["zeta"] = 5e-5
    tab = mlpol.Tables(atom)
    x = mlpol.lte_unknowns(tab, atm["kT"])
    rng = np.random.default_rng(m)
    rb = mlpol.real_basis(atom)
    for k, (i, K, Q, part) in enumerate(rb):
        if K > 0:
            x[..., k] = 0.02 * x[..., rb.index((i, 0, 0, 0))] * rng.normal(size=x.shape[:-1])
    got = []
    for solve in (0, 1):
        c = P.MlContext(atm, atom, 2, 4, 5, precision=P.PORTA_FP64, polarized=True)
        c.set_atmosphere(atm)
        c.set_unknowns(x)
        c.set_solve(solve)
        c.ml_iterate(1)
        got.append(c.get_unknowns())
    assert np.max(np.abs(got[0] - got[1])) < 1e-11 * np.max(np.abs(got[1]))
    assert np.max(np.abs(got[0] - x)) > 1e-6
