"""The division (||Y||_F^2 - Tr P) / N of a layer's offset, replayed on the CPU: on the device
it is a product with the rounded reciprocal 1/N and one residual step (two FMAs).  The result
has to be the correctly rounded quotient for every N up to 65536, as a division gives it."""
import math
import random
from fractions import Fraction


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # one rounding, to nearest even


def device_quotient(dev, n):
    inv = 1.0 / n
    g0 = dev * inv
    return fma(fma(-g0, float(n), dev), inv, g0)


def test_offset_quotient_is_correctly_rounded():
    rng = random.Random(5)
    sizes = [1, 2, 3, 5, 7, 127, 129, 1537, 4095, 4097, 65535, 65536] + [rng.randint(1, 65536) for _ in range(300)]
    # Sizes whose reciprocal rounds worst, where the first quotient is furthest off.
    sizes += sorted(range(3, 65536, 7), key=lambda n: -abs(Fraction(1.0 / n) * n - 1))[:40]
    off = 0
    for n in sizes:
        for _ in range(60):
            mantissa = rng.choice([rng.random() + 1.0, 2.0 - rng.randint(1, 99) * 2.0 ** -52, 1.0 + rng.randint(0, 99) * 2.0 ** -52])
            dev = rng.choice([-1.0, 1.0]) * math.ldexp(mantissa, rng.randint(-60, 20))
            assert device_quotient(dev, n) == dev / n
            off += dev * (1.0 / n) != dev / n
        assert device_quotient(0.0, n) == 0.0
    assert off > 1000   # the first quotient alone is not
