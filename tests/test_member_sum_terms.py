"""The member sums' terms g(n-1), g(n), g(n+1) of one member, as the kernel
computes them, against exact rationals.  k (k-1) and (d-1)(D+1) are integers;
below 2^53 both are exact in FP64, so each term has to be the correctly rounded
quotient; above, the two products and the quotient round once each."""
import ctypes as C
from fractions import Fraction as Fr

import numpy as np
import pytest

from device_source import build

U64 = Fr(1, 2 ** 53)


@pytest.fixture(scope="module")
def g3(tmp_path_factory):
    lib = build(tmp_path_factory.mktemp("g3"), ["lit_g3"], [], """
extern "C" void g3(int32_t k, int32_t d, int32_t n, double *f) { lit_g3(k, d, n, f[0], f[1], f[2]); }
""")

    def call(k, d, n):
        f = (C.c_double * 3)()
        lib.g3(k, d, n, f)
        return [f[0], f[1], f[2]]
    return call


def exact(k, d, nu):
    return Fr(k * (k - 1), (d - 1) * (nu - 1 + d - k)) if k >= 2 and d >= 2 else Fr(0)


@pytest.mark.parametrize("top", [4, 40, 3000, 40000, 1 << 20, 1 << 26, 1 << 30])
def test_terms_are_rounded_as_little_as_fp64_allows(g3, top):
    rng = np.random.default_rng(top)
    for _ in range(3000):
        d = int(rng.integers(1, top))
        n = int(rng.integers(2, top))
        k = int(rng.integers(0, min(d, n - 1) + 1))   # a member's neighbours inside
        D = n - 1 + d - k
        once = k * (k - 1) < 2 ** 53 and (d - 1) * (D + 1) < 2 ** 53
        for got, nu in zip(g3(k, d, n), (n - 1, n, n + 1)):
            want = exact(k, d, nu)
            if once:
                assert got == float(want), (k, d, n, nu)
            else:
                assert abs(Fr(got) - want) <= ((1 + U64) ** 2 / (1 - U64) - 1) * want, (k, d, n, nu)
