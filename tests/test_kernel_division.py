"""The kernels' division by a known reciprocal, in exact arithmetic on the CPU.

div_by(a, b, fl(1/b)) estimates a / b as fl(a rb) and corrects it twice by its
exact remainder, fl(q + fl(a - b q) rb).  Checked against the correctly rounded
quotient (rational arithmetic, one rounding) over random operands, operands
whose quotients lie next to rounding boundaries, and the divisors the kernels
use (10,000 for depths, focal lengths, vertex depths)."""
from fractions import Fraction

import numpy as np


def _round32(x: Fraction) -> Fraction:
    """x rounded to 24 significant bits, ties to even (no overflow or underflow)."""
    if x == 0:
        return x
    n, d = abs(x.numerator), x.denominator
    e = n.bit_length() - d.bit_length()
    if Fraction(n, d) < Fraction(2) ** e:
        e -= 1
    scale = Fraction(2) ** (23 - e)
    m = abs(x) * scale
    lo = m.numerator // m.denominator
    r = m - lo
    lo += r > Fraction(1, 2) or (r == Fraction(1, 2) and lo % 2 == 1)
    return (1 if x > 0 else -1) * lo / scale


def _div_by(a: Fraction, b: Fraction) -> Fraction:
    rb = _round32(1 / b)
    q = _round32(a * rb)
    for _ in range(2):
        q = _round32(q + _round32(a - b * q) * rb)
    return q


def test_two_corrections_give_the_rounded_quotient():
    rng = np.random.default_rng(3)
    a = [float(np.float32(x)) for x in rng.uniform(-4, 4, 4000) * 2.0 ** rng.integers(-40, 40, 4000)]
    b = [float(np.float32(x)) for x in rng.uniform(0.5, 1, 4000) * 2.0 ** rng.integers(-40, 40, 4000)]
    # significands all ones, one above a power of two, and small ones
    edge = [1.0, float(np.nextafter(np.float32(2), np.float32(0))), float(np.nextafter(np.float32(1), np.float32(2))), 3.0]
    a += [x * y for x in edge for y in (1.0, -1.0, 2.0 ** -59, 2.0 ** 59)] * 4
    b += [x for x in edge for _ in range(16)]
    # depths in 0.1 mm units, and products of pixel offsets and depths over a focal length
    a += [float(d) for d in rng.integers(1, 65536, 2000)] + [0.0]
    b += [10000.0] * 2001
    a += [float(np.float32(u) * np.float32(z)) for u, z in zip(rng.integers(-640, 640, 2000) + 0.5, rng.uniform(0.05, 6.5, 2000))]
    b += [615.0, 150.0, 307.5, 571.3999633789062] * 500
    # quotients a hair from a rounding boundary: a next to b (q + half a unit)
    for _ in range(2000):
        y = np.float32(rng.uniform(0.5, 2))
        q = np.float32(rng.uniform(0.5, 2))
        half = (Fraction(float(q)) + Fraction(float(np.nextafter(q, np.float32(4))))) / 2
        b.append(float(y))
        a.append(float(_round32(half * Fraction(float(y)))))
    assert len(a) == len(b)
    for x, y in zip(a, b):
        x, y = Fraction(x), Fraction(y)
        assert _div_by(x, y) == _round32(x / y), (float(x), float(y))
