"""The two-limb fixed-point sums of the f64 tensor-core path's per-row kernels (csrc/fixed.cuh and key_exps
in csrc/tab_gemm.cuh), restated in exact integers: no accumulator leaves 63 bits at the operands' bounds,
and every result lies within the stated units of the exact value (CPU)."""
import math
from fractions import Fraction as Fr

import numpy as np
import pytest

PLACES, L = 61, 30  # of the rows kernel


def limbs(v, b):
    return v >> b, v & ((1 << b) - 1)


def acc(terms, b):
    hi = mid = 0
    for x, y in terms:
        (xh, xl), (yh, yl) = limbs(x, b), limbs(y, b)
        assert max(abs(xh), abs(yh)) <= 1 << 31 and max(xl, yl) < 1 << 31
        hi += xh * yh
        mid += xh * yl + xl * yh
        assert abs(hi) < 1 << 63 and abs(mid) < 1 << 63
    return hi, mid


def over_unit(p, b):
    hi, mid = p
    mid += 1 << (b - 1)
    assert abs(mid) < 1 << 63
    return hi + (mid >> b)


def mul(x, y, b):
    return over_unit(acc([(x, y)], b), b)


def key_exps(E, e):
    a = [E[q] - e * q for q in range(6)]
    top = max(a[1:])
    s = sum(((q << 20) >> min(top - a[q], 31)) + 1 for q in range(1, 6))
    assert s < 1 << 24
    slope = top - 20 + s.bit_length()
    return max(a[0], slope) + 1, slope


@pytest.mark.parametrize("case", ["smooth", "flat", "high order", "signs", "one term"])
def test_row_polynomial(case):
    """P = d_0 + sum D_q u^q / q and P' = sum D_q u^(q-1) against exact rationals, over u in [-1e-4, 1/1.05]: the
    products' dropped limbs, the powers' truncation and the two roundings stay below 16 units of 2^(X + G - 61)
    (five terms: each at most 1 + 2 units from its product and power, and the roundings)."""
    rng = np.random.default_rng(7)
    E = {"smooth": [1, -5, -12, -18, -25, -33], "flat": [2] * 6, "high order": [0, -9, -7, -4, -2, 0],
         "signs": [0, -1, 0, -1, 0, -1], "one term": [-900, 3, -900, -900, -900, -900]}[case]
    G = 7
    value, slope = key_exps(E, 0)
    worst = [0.0, 0.0]
    for it in range(400):
        edge = it % 4 == 0
        d = [Fr(int((1 if edge else rng.random()) * rng.choice([-1, 1]) * (2**53 - 1)), 2**53) * Fr(2) ** (E[q] + G)
             for q in range(6)]
        u = Fr(int(rng.choice([0.0, 1 / 1.05, -1e-4, rng.random() / 1.05]) * 2**60), 2**60)
        uq = [None, int(u * 2**60)]
        uq.append(mul(uq[1], uq[1], L))
        uq.append(mul(uq[2], uq[1], L))
        uq.append(mul(uq[2], uq[2], L))
        u5 = mul(uq[4], uq[1], L)
        w = [None, uq[1], uq[2] >> 1, mul(uq[3], (0x15555555 << 30) + 0x15555555, L), uq[4] >> 2,
             mul(u5, (0x0ccccccc << 30) + 0x33333333, L)]
        D = [round(q * d[q] / Fr(2) ** (slope + G - PLACES)) for q in range(6)]
        d0 = round(d[0] / Fr(2) ** (value + G - PLACES))
        assert sum(abs(x) for x in D) < 1 << PLACES
        p = over_unit(acc([(D[q], w[q]) for q in range(1, 6)], L), L)
        g = D[1] + over_unit(acc([(D[q], uq[q - 1]) for q in range(2, 6)], L), L)
        P = d0 + (p >> (value - slope))
        assert abs(P) < 1 << 62 and abs(g) < 1 << 62
        ex = sum(d[q] * u**q for q in range(6)) / Fr(2) ** (value + G - PLACES)
        eg = sum(q * d[q] * u ** (q - 1) for q in range(1, 6)) / Fr(2) ** (slope + G - PLACES)
        worst = [max(worst[0], abs(float(P - ex))), max(worst[1], abs(float(g - eg)))]
    assert max(worst) <= 16.0, worst


def test_moment_sums():
    """32 rows of the largest R~ (57 places) times powers of u up to 1.125 (56 places): no overflow, and each sum
    within 2 units a row of the exact one (a truncated R~, a truncated power, the dropped limb product)."""
    b = 28
    rng = np.random.default_rng(3)
    for it in range(60):
        r = [Fr(int(x)) for x in (rng.choice([-1, 1], 32) * (2**57 - 1 - rng.integers(0, 2**50 * (it % 2) + 1, 32)))]
        u = Fr(int(rng.choice([1.0, 1.0001, rng.random()]) * 2**53), 2**53)
        u1 = int(u * 2**56)
        u2 = mul(u1, u1, b)
        u3 = mul(u2, u1, b)
        powers = [1 << 56, u1, u2, u3, mul(u2, u2, b), mul(u3, u2, b)]
        for q in range(6):
            got = over_unit(acc([(int(x), powers[q]) for x in r], b), b)
            # the power's own error (at most q + 1 units of 2^-56) times R~ < 2^57, and the dropped limbs
            assert abs(got - sum(r) * u**q) <= 32 * (2 * (q + 1) + 1)
            assert abs(got) < 1 << 63


def test_bounds_hold():
    """2^slope exceeds the derivative's coefficients' sum and 2^value every part of the polynomial."""
    rng = np.random.default_rng(11)
    for _ in range(500):
        E, e = [int(x) for x in rng.integers(-60, 20, 6)], int(rng.integers(-3, 12))
        value, slope = key_exps(E, e)
        a = [Fr(2) ** (E[q] - e * q) for q in range(6)]
        assert sum(q * a[q] for q in range(1, 6)) < Fr(2) ** slope
        assert a[0] <= Fr(2) ** (value - 1) and slope < value
        assert math.log2(float(sum(q * a[q] for q in range(1, 6)))) > slope - 2


def _constants():
    """The switch's coefficient tables, from the source."""
    import os
    import re
    src = open(os.path.join(os.path.dirname(__file__), "..", "paper_2107_02103_gb300", "csrc", "env_row.cuh")).read()
    return [[int(x) for x in re.search(rf"{n}\[12\] = {{(.*?)}}", src, re.S).group(1).split(",")] for n in ("kSin", "kCos")]


@pytest.mark.parametrize("kind", [0, 1])
def test_switch(kind):
    """The weighting function and its derivative in fixed point against 60-digit arithmetic over u in [0, 1]: within
    2^-55 and 2^-53 (eleven Horner steps each off by at most two units of 2^-60, over 4; their last powers' sum)."""
    from decimal import Decimal as Dc, getcontext
    getcontext().prec = 60
    pi = Dc("3.14159265358979323846264338327950288419716939937510582097494459")

    def series(x, first):  # sin (first = 1) or cos (first = 0) of x
        term = x if first else Dc(1)
        total, n = term, first
        while abs(term) > Dc(10) ** -50:
            term *= -x * x / ((n + 1) * (n + 2))
            total += term
            n += 2
        return total

    ksin, kcos = _constants()
    rng = np.random.default_rng(2)
    for uf in [0.0, 2.0 ** -60, 1e-9, 0.5, 1 - 2.0 ** -53, 1.0, *rng.random(200)]:
        u = int(Fr(uf) * 2**60)
        U = Dc(u) / Dc(2) ** 60
        if kind == 1:
            u2 = mul(u, u, L)
            u3 = mul(u2, u, L)
            q8 = (2 * u - (u >> 3)) - (u2 - (u2 >> 2)) - (5 << 58)
            w, dw = (1 << 60) + 8 * mul(u3, q8, L), -(15 * mul(u2 - u, u2 - u, L) >> 1)
            ew, ed = U**3 * (-6 * U * U + 15 * U - 10) + 1, -30 * U * U * (U - 1) ** 2
        else:
            x = u - (1 << 59)
            z = mul(x, x, L)
            p, q = ksin[11], kcos[11]
            for k in range(10, -1, -1):
                p, q = ksin[k] + mul(p, z, L), kcos[k] + mul(q, z, L)
                assert max(abs(p), abs(q)) < 1 << 61
            w, dw = (1 << 59) - 2 * mul(p, x, L), -q
            ew, ed = series(pi * U, 0) / 2 + Dc("0.5"), -(pi / 2) * series(pi * U, 1)
        assert abs(w) < 1 << 62 and abs(Dc(w) / Dc(2) ** 60 - ew) < Dc(2) ** -55
        assert abs(Dc(dw) / Dc(2) ** 58 - ed) < Dc(2) ** -53
