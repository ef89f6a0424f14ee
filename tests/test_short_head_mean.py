"""The K channel mean of short heads, sum / n in three operations with 1 / n at hand (divided() in vc_prep.cu), is the quotient
correctly rounded for every token count of a cluster's blocks."""
import random
from fractions import Fraction

import pytest

TOKENS = 1024            # blocks of 128 tokens, eight at most


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))       # (a Fraction is rounded to nearest even)


def _divided(x, n, inv):
    q = x * inv
    return _fma(_fma(-q, n, x), inv, q)


@pytest.mark.parametrize("first", range(1, TOKENS + 1, 128))
def test_is_the_quotient(first):
    rng = random.Random(first)
    for n in range(first, first + 128):
        inv = 1.0 / n
        for _ in range(24):
            x = rng.uniform(-1.0, 1.0) * 2.0 ** rng.randint(-140, 130)
            # the sums nearest to n times a number halfway between two doubles, where the rounding is decided
            k = rng.randrange(2 ** 52, 2 ** 53)
            halfway = float(Fraction(2 * k + 1, 2) * n)
            for s in (x, halfway, -halfway, float(n * k)):
                assert _divided(s, float(n), inv) == s / n, (s, n)
