"""The one expression the bracket uses for a neighbour's correction when x joins or
leaves a community, emulated in float32 operation by operation and compared with
the difference of the two estimators in exact rationals: at most five roundings
for arguments below 2^24 (conversions and the decrements are exact there), so a
relative error below (1 + 2^-24)^5 - 1 and zero exactly where the difference is."""
from fractions import Fraction as Fr

import numpy as np
import pytest

f32 = np.float32


def h32(own, k, d, n):
    if d < 2 or k < (2 if own else 1) or (own and n < 3):
        return f32(0)
    e, kk = f32(n + (d - k) - (1 if own else 0)), f32(k - 1 if own else k)
    num = f32(kk * f32(f32(2) * e + f32(kk - f32(1))))
    h = f32(num / f32(f32(d - 1) * f32(e * f32(e - f32(1)))))
    return -h if own else h


def g(k, d, nu):
    return Fr(k * (k - 1) * d, d * (d - 1)) / (nu - 1 + d - k) if k >= 2 and d >= 2 else Fr(0)


def exact(own, k, d, n):
    if own:     # y stays in C, x leaves: size n - 1, one neighbour fewer
        return g(k - 1, d, n - 1) - g(k, d, n - 1) if n >= 3 and k >= 1 else Fr(0)
    return g(k + 1, d, n + 1) - g(k, d, n + 1)


@pytest.mark.parametrize("own", [False, True])
@pytest.mark.parametrize("top", [6, 200, 40000, 1 << 23])
def test_correction_rounding(own, top):
    rng = np.random.default_rng(top + own)
    bound = (1 + Fr(1, 2 ** 24)) ** 5 - 1
    for _ in range(2000):
        d = int(rng.integers(1, top))
        n = int(rng.integers(2, top))
        k = int(rng.integers(0, min(d - (0 if own else 1), n - 1 if own else n) + 1))   # x is a neighbour of y too
        got, want = Fr(float(h32(own, k, d, n))), exact(own, k, d, n)
        assert abs(got - want) <= bound * abs(want), (own, k, d, n)
