"""The quotient by the temperature that the fused pass forms without a division: its steps, restated in exact arithmetic with every
rounding made explicit, against the correctly rounded quotient over the range that the pass claims for them."""
import math
from fractions import Fraction

import numpy as np
import pytest

TINY, HUGE = Fraction(1, 2 ** 149), Fraction(2) ** 128


def fl(x: Fraction) -> Fraction:
    """x rounded to fp32 (to nearest, ties to even; subnormal numbers kept)."""
    if x == 0:
        return x
    m = abs(x)
    e = m.numerator.bit_length() - m.denominator.bit_length()
    if m < Fraction(2) ** e:
        e -= 1
    unit = max(Fraction(2) ** (e - 23), TINY)
    q, r = divmod(m, unit)
    q += 1 if 2 * r > unit or (2 * r == unit and q % 2) else 0
    assert q * unit < HUGE
    return q * unit if x > 0 else -q * unit


def divisor(T: Fraction):
    """What the host passes: 1 / T rounded, and rounded towards zero with what that leaves (the reciprocal itself is a double there)."""
    inv = Fraction(1.0 / float(T))
    y = fl(inv)
    hi = Fraction(float(np.nextafter(np.float32(float(y)), np.float32(0)))) if y > inv else y
    lo = fl(inv - hi)
    return y, hi, lo if lo > 0 else Fraction(1, 2 ** 126)


def quotient(x: Fraction, T: Fraction, y, hi, lo):
    q = fl(x * hi + fl(x * lo))
    return fl(fl(x - q * T) * y + q)


TEMPERATURES = [0.5, 0.7, 0.9, 1.2, 3.0, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -23, 1.0 / 3.0, 1e-3, 1e3, 1.2e-30, 1.2e30, 2.0 ** -100, 2.0 ** 100,
                float.fromhex("0x1.8p99"), float.fromhex("0x1.fffffep-100")]


@pytest.mark.parametrize("T", TEMPERATURES)
def test_quotient_is_the_divisions(T):
    T = Fraction(float(np.float32(T)))
    host = divisor(T)
    rng = np.random.default_rng(3)
    least = max(Fraction(1, 2 ** 100), T / 2 ** 125)              # the smallest logit the steps are claimed for
    most = min(HUGE, HUGE * T) / 4
    e0, e1 = math.ceil(math.log2(least)), math.floor(math.log2(most))
    exps = np.concatenate([rng.integers(e0, e1, 250), np.full(150, e0), np.clip(rng.integers(-8, 8, 150), e0, e1 - 1)])
    near = np.concatenate([rng.integers(0, 2 ** 23, exps.size - 40), np.arange(20), 2 ** 23 - 1 - np.arange(20)])
    for e, m in zip(exps, near):
        x = (1 + Fraction(int(m), 2 ** 23)) * Fraction(2) ** int(e)
        if x < least:
            continue
        assert quotient(x, T, *host) == fl(x / T), (float(x), float(T))
        assert quotient(-x, T, *host) == fl(-x / T)
    assert quotient(Fraction(0), T, *host) == 0


def test_below_that_the_remainder_is_lost():
    """Why the pass looks for smaller logits where the very value matters: some are off by a unit in the last place."""
    T = Fraction(float(np.float32(0.9)))
    host, rng, off = divisor(T), np.random.default_rng(4), 0
    for m in rng.integers(0, 2 ** 23, 500):
        x = (1 + Fraction(int(m), 2 ** 23)) / 2 ** 125
        off += quotient(x, T, *host) != fl(x / T)
    assert off
