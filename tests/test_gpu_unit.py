"""The step coefficients and the profile as the J^K_Q sweep evaluates them, against 40-digit
evaluations of the closed forms.

FP32, two frequencies at a time, the pairs' lanes mostly on different sides of t = 1.5, where
polynomials give way to closed forms. A unit of rounding is 6e-8. e0 = 1 - e^-t: two roundings of
t (1 - h). w_M, w_O: a polynomial of relative error 5e-9 and its last two roundings, or a closed form
that multiplies three roundings by up to 3. w_C = e0 - w_M - w_O below 1.5, where it is at least a
quarter of e0, so that the roundings of the three weigh up to 4 times: 8e-7; w_O + w_C = e0 - w_M, at
least 0.6 of e0: 3e-7. e^-t = 1 - e0 to a rounding, absolutely. The profile: the exponent's three
roundings are 1.8e-7 of x^2, the approximation of 2^y adds 2.4e-7.

FP64: a polynomial of degree 12 or a closed form in e0 that loses a factor of up to 10 to
cancellation: 5e-15, a few points on either side of t = 1 among them. The profile: a table entry
(2^-52), the last rounding (2^-53) and the polynomial and argument (1e-16) on a given x^2: 4.5e-16.
"""
import mpmath
import numpy as np
import pytest

import paper_1307_4217_gb300 as P

pytestmark = pytest.mark.gpu


def _exact(t):
    t = mpmath.mpf(float(t))
    e = mpmath.exp(-t)
    return [e, 1 - e, (2 - e * (t * t + 2 * t + 2)) / t**2, 1 - 2 * (e + t - 1) / t**2, 2 * (t - 2 + e * (t + 2)) / t**2]


def _run(prec, t, x):
    mpmath.mp.dps = 40
    rc, out = P.porta_eval_unit(prec, t, x)
    assert rc == P.PORTA_OK
    return out, [_exact(v) for v in t]


def _rel(a, b):
    return float(abs((mpmath.mpf(float(a)) - b) / b))


def test_fp32():
    rng = np.random.default_rng(1)
    t = rng.permutation(np.geomspace(1e-7, 1e3, 2001)).astype(np.float32).astype(np.float64)
    t[:8] = np.float32([1.4999999, 1.5, 1.5, 1.4999999, 1e-7, 1e3, 1e3, 1e-7])
    x = rng.permutation(np.linspace(-6, 6, len(t))).astype(np.float32).astype(np.float64)
    out, ex = _run(P.PORTA_FP32, t, x)
    for o, r, v in zip(out, ex, x):
        assert abs(float(o[0] - r[0])) < 1.8e-7 and abs(o[0] + o[1] - 1) <= 6e-8
        assert _rel(o[1], r[1]) < 1.8e-7
        assert _rel(o[2], r[2]) < 6e-7 and _rel(o[3], r[3]) < 6e-7
        assert _rel(o[4], r[4]) < 8e-7
        assert _rel(np.float32(o[3]) + np.float32(o[4]), r[3] + r[4]) < 3.6e-7
        assert _rel(o[5], mpmath.exp(-mpmath.mpf(v) ** 2)) < 2.4e-7 + 1.8e-7 * v * v


def test_fp64():
    rng = np.random.default_rng(2)
    t = np.concatenate([np.geomspace(1e-7, 1e3, 2001), 1 + np.arange(-4, 5) * 2.0**-52, [0.999, 1.001]])
    x = rng.permutation(np.concatenate([np.linspace(-25, 25, len(t) - 2), [0.0, 1e-9]]))
    out, ex = _run(P.PORTA_FP64, t, x)
    for o, r, v in zip(out, ex, x):
        for k in range(1, 5):
            assert _rel(o[k], r[k]) < 5e-15
        assert abs(float(o[0] - r[0])) < 2.3e-16 + 5e-15 * float(r[0])
        assert _rel(o[5], mpmath.exp(-mpmath.mpf(v * v))) < 4.5e-16
