"""The quotient of two FP32 pairs by which the resident FP32 PCG forms alpha and beta, restated in numpy
with single roundings, against the exact one: as near to it as the FP64 quotient rounded to FP32."""
from fractions import Fraction

import numpy as np

F = np.float32


def _pair(v):
    hi = F(v)
    return hi, F(v - float(hi))


def _over(s, e, ds, de):
    q = F(s / ds)
    exact = float(s) - float(q) * float(ds)  # the fma: exact here, rounded once
    r = F(F(exact) + F(e - F(q * de)))
    return F(q + F(r / ds))


def test_quotient_is_rounded_once():
    rng = np.random.default_rng(5)
    worst, worst64, differ = 0.0, 0.0, 0
    n = 20000
    for _ in range(n):
        x, y = (float(rng.uniform(1, 2) * 2.0 ** rng.integers(-30, 30)) for _ in range(2))
        (s, e), (ds, de) = _pair(x), _pair(y)
        exact = Fraction(float(s)) + Fraction(float(e))
        exact /= Fraction(float(ds)) + Fraction(float(de))
        got = _over(s, e, ds, de)
        f64 = F((float(s) + float(e)) / (float(ds) + float(de)))
        ulp = Fraction(float(np.spacing(abs(f64))))
        worst = max(worst, float(abs(Fraction(float(got)) - exact) / ulp))
        worst64 = max(worst64, float(abs(Fraction(float(f64)) - exact) / ulp))
        differ += int(got != f64)
    # half an ulp and what the correction leaves out, 2^-23 of its own half ulp
    assert worst64 <= 0.5 + 1e-6 and worst <= 0.5 + 1e-6
    assert differ <= 2  # ties to a few parts in 10^7 only
