"""The fitting net's digit scheme on the tensor cores (eight balanced 7-bit digits, the 36 products with s + t <= 9,
512 of K per exact share), emulated exactly as in test_digit_split, and its recombination in 64-bit words (CPU)."""
from fractions import Fraction

import numpy as np
import pytest

from test_digit_split import product

SCHEME_8x7 = (8, 7, 55, sum(64 * 128 ** k for k in range(7)), 512, -50)


@pytest.mark.parametrize("K,scaled", [(1, False), (70, False), (512, False), (513, False), (40, True)])
def test_digit_product_within_its_bound(K, scaled):
    rng = np.random.default_rng(K)
    A, B = rng.standard_normal((3, K)), rng.standard_normal((K, 2))
    if scaled:
        A *= 10.0 ** rng.uniform(-30, 30, (3, 1))
        A[0] = 0.0
        A[1, ::3] = 0.0
    C, peak = product(A, B, SCHEME_8x7)
    assert peak <= 2 ** 24
    for i in range(3):
        for j in range(2):
            exact = sum(Fraction(A[i, k]) * Fraction(B[k, j]) for k in range(K))
            bound = K * 2.0 ** -50 * np.abs(A[i]).max() * np.abs(B[:, j]).max()
            assert abs(Fraction(C[i, j]) - exact) <= Fraction(bound) + Fraction(abs(float(exact))) * 2 ** -52


def test_exactness_at_the_extremes():
    """Every digit at the end of its range: a diagonal's sum over a share is at most 2^24, which fp32 holds, and
    the two parts of the recombined integer are exact in 64 bits and as doubles."""
    assert 8 * 64 * 64 * 512 == 2 ** 24
    for sign in (1, -1):
        x = [sign * min(d + 1, 8) * 64 * 64 * 512 for d in range(8)]
        T, M, low = x[0] * 16384 + x[1] * 128 + x[2], x[3] * 16384 + x[4] * 128 + x[5], x[6] * 128 + x[7]
        A = M * 16384 + low
        assert abs(T) < 2 ** 53 and abs(A) <= 2 ** 53 and float(T) == T and float(A) == A
        assert (T << 35) + A == sum(v << (7 * (7 - d)) for d, v in enumerate(x))
