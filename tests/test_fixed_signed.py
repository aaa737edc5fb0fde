"""The limb sums with signed low limbs (csrc/fixed.cuh), restated in exact integers (CPU): at the operands' bounds of each
kernel no accumulator leaves 63 bits and no limb 32, every sum is within its stated units, and the errors of many sums
have no common sign."""
import random

import pytest


def limbs(v, b):
    hi = (v + (1 << (b - 1))) >> b
    lo = v - (hi << b)
    assert -(1 << 31) <= hi < 1 << 31 and -(1 << (b - 1)) <= lo < 1 << (b - 1)
    return hi, lo


def total(terms, b, start=0):
    hi, mid = start, 0
    for x, y in terms:
        (xh, xl), (yh, yl) = limbs(x, b), limbs(y, b)
        hi += xh * yh
        mid += xh * yl + xl * yh
        assert abs(hi) < 1 << 63 and abs(mid) < 1 << 63
    mid += 1 << (b - 1)
    out = hi + (mid >> b)
    assert abs(mid) < 1 << 63 and abs(out) < 1 << 63
    return out


# terms, places of either factor, limb: D, the descriptor's backward, the moments (powers of u up to 1.125)
@pytest.mark.parametrize("n,p,q,b", [(4, 60, 60, 30), (16, 57, 57, 28), (32, 57, 56.17, 28)])
def test_sums_at_the_bounds(n, p, q, b):
    rng = random.Random(n)
    P, Q = int(2 ** p), int(2 ** q)  # (a conversion to nearest can reach the power itself)
    for it in range(2000):
        if it < 16:  # every sign, the extremes
            xs, ys = [P if it & 1 else -P] * n, [Q if it & 2 else -Q] * n
            if it & 4:
                xs[0] = P - rng.randrange(1 << b)
            if it & 8:
                ys[-1] = -(1 << (b - 1)) - (1 << b)
        else:
            xs, ys = [rng.randint(-P, P) for _ in range(n)], [rng.randint(-Q, Q) for _ in range(n)]
        got, want = total(zip(xs, ys), b) << (2 * b), sum(x * y for x, y in zip(xs, ys))
        # a quarter of a unit from each dropped product, half from the rounding
        assert abs(got - want) <= (n + 2) << (2 * b - 2)


def test_zeros_and_signs():
    assert total([(0, 12345)] * 5, 30) == 0 and total([(1 << 59, 0)], 30) == 0
    rng = random.Random(1)
    err = []
    for _ in range(20000):
        xs, ys = [rng.randint(-2 ** 59, 2 ** 59) for _ in range(4)], [rng.randint(-2 ** 59, 2 ** 59) for _ in range(4)]
        err.append((total(zip(xs, ys), 30) * 2 ** 60 - sum(x * y for x, y in zip(xs, ys))) / 2 ** 60)
    mean, rms = sum(err) / len(err), (sum(e * e for e in err) / len(err)) ** 0.5
    assert abs(mean) <= 5 * rms / len(err) ** 0.5


@pytest.mark.parametrize("drop", range(0, 32))
def test_the_rows_half(drop):
    """The slope's sum enters the value's units rounded, not floored: half = 2^drop / 2 added before the shift."""
    half = (1 << drop) >> 1
    for v in (0, 1, -1, (1 << 61) - 1, -(1 << 61) + 1, 3 << max(drop - 1, 0), -(3 << max(drop - 1, 0))):
        assert abs(((v + half) >> drop) * (1 << drop) - v) * 2 <= 1 << drop
    assert (0 + half) >> drop == 0
