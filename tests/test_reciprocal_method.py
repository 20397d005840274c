"""The reciprocal of the training kernel's sigmoids: one step of the
Newton-Raphson iteration y (2 - d y) = y + y (1 - d y), as two fused
multiply-adds, on an approximation within one unit in the last place (what PTX
states for rcp.approx.ftz.f32).  Checked on the CPU in exact rational
arithmetic: within 0.51 units in the last place for every approximation that
close, over the denominators 1 + e^-z with z from -80 on."""
import math
from fractions import Fraction

import numpy as np


def _ulp(x: Fraction) -> Fraction:
    return Fraction(2) ** (math.frexp(float(x))[1] - 24)


def _rn(x: Fraction) -> Fraction:
    """x rounded to nearest, ties to even, in FP32 (normal range)."""
    if x == 0:
        return x
    u = _ulp(abs(x))
    return round(x / u) * u


def test_one_newton_step_from_a_close_approximation():
    rng = np.random.default_rng(1)
    z = np.concatenate([rng.uniform(-80.0, 20.0, 1500), rng.normal(0.0, 3.0, 1500)])
    ds = np.concatenate([(1.0 + np.exp(-z)).astype(np.float32),
                         [1.0, 2.0, np.nextafter(np.float32(2), np.float32(0)), np.nextafter(np.float32(1), np.float32(2)),
                          np.float32(2.0) ** 115, np.nextafter(np.float32(2.0) ** 115, np.float32(0))]])
    worst = Fraction(0)
    for d in ds.tolist():
        d = Fraction(d)
        for step in (-1, 0, 1):
            y = _rn(1 / d) + step * _ulp(1 / d)
            if abs(y - 1 / d) > _ulp(1 / d):
                continue   # further off than the approximation may be
            e = _rn(1 - d * y)          # fma(-d, y, 1)
            y = _rn(e * y + y)          # fma(e, y, y)
            worst = max(worst, abs(y - 1 / d) / _ulp(1 / d))
    assert worst <= Fraction(51, 100), float(worst)
