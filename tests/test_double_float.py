"""Double-float differences in binary32 on the CPU: the error that the screen's bounds allow for."""
from fractions import Fraction

import numpy as np
import pytest

f32 = np.float32


def _difference(v, d):
    """d - v as the y preparation forms it: v as hi + lo, TwoSum of hi and -d, and lo added once."""
    hi = f32(v)
    lo = f32(np.float64(v) - np.float64(hi))
    s = f32(hi - d)
    bb = f32(s - hi)
    e = f32(f32(hi - f32(s - bb)) + f32(f32(-d) - bb))
    return -f32(s + f32(e + lo))


@pytest.mark.parametrize("scale", [1e-3, 1.0, 300.0, 1e6])
def test_difference_within_three_quarters_of_a_unit(scale):
    """|error| <= 1.5 2^-24 |d - v| (and second-order terms), for data at, next to, and far from the centre."""
    rng = np.random.default_rng(int(scale) + 1)
    worst = Fraction(0)
    for _ in range(4000):
        v = np.float64(scale * rng.uniform(0.4, 2.1))
        if rng.random() < 0.3:  # the low half just below and above half a unit of the high one
            h = f32(v)
            v = np.float64(h) + np.float64(np.spacing(h)) * (0.5 + rng.uniform(-1, 1) * 2.0 ** -rng.integers(1, 29))
        hi = f32(v)
        k = int(rng.integers(-3, 4))
        d = {0: f32(hi + k * np.spacing(hi)), 1: f32(hi * rng.uniform(0.5, 2.0)), 2: f32(rng.integers(0, 2000))}[
            int(rng.integers(0, 3))]
        exact = Fraction(float(d)) - Fraction(float(v))
        got = Fraction(float(_difference(v, d)))
        if exact == 0:
            assert got == 0
            continue
        worst = max(worst, abs(got - exact) / abs(exact))
    assert worst <= Fraction(3, 2) * Fraction(1, 2 ** 24) * (1 + Fraction(1, 2 ** 20))
    assert worst > Fraction(1, 2 ** 25)  # the bound is met within a factor of a few
