"""The quotients formed from a reciprocal (tile test, transmittance
restoration) round as the general division does; float32 arithmetic in exact
rationals, on the CPU."""
from fractions import Fraction

import numpy as np
import pytest


def _rn(x: Fraction) -> np.float32:
    """x rounded to float32, ties to even."""
    f = np.float32(float(x))  # within an ulp; pick the nearest of three
    best = None
    for c in (np.nextafter(f, np.float32(-np.inf)), f, np.nextafter(f, np.float32(np.inf))):
        d = abs(Fraction(float(c)) - x)
        even = (int(c.view(np.uint32)) & 1) == 0
        if best is None or d < best[0] or (d == best[0] and even):
            best = (d, c)
    return best[1]


def _fma(a, b, c):
    return _rn(Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c)))


def _div_recip(n, d, y):
    q = _rn(Fraction(float(n)) * Fraction(float(y)))
    return _fma(_fma(-d, q, n), y, q)


@pytest.mark.parametrize("kind", ["tile", "transmittance"])
def test_corrected_quotient_is_the_rounded_one(kind):
    rng = np.random.default_rng(0)
    for _ in range(3000):
        if kind == "tile":
            d = np.float32(2.0 ** rng.uniform(-40, 5))
            n = np.float32(rng.choice([-1, 1]) * 2.0 ** rng.uniform(-60, 20))
            y = _rn(1 / Fraction(float(d)))
        else:
            d = np.float32(1) - np.float32(min(0.99, 2.0 ** rng.uniform(-8, 0)))
            n = np.float32(2.0 ** rng.uniform(-13.3, 0))
            r = _rn(1 / Fraction(float(d)))
            for _ in range(rng.integers(0, 3)):  # the approximate reciprocal: up to 2 ulp off
                r = np.nextafter(r, np.float32(rng.choice([0.0, 4.0])))
            y = _fma(_fma(-d, r, np.float32(1)), r, r)
        assert _div_recip(n, d, y) == _rn(Fraction(float(n)) / Fraction(float(d))), (n, d)
