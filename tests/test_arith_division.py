"""Host check of the split kernels' FP64 quotient from a reciprocal, for sums
that are no integers, against exact rational arithmetic: with inv = RN(1 / b),
q0 = RN(s inv), the exact residual r = s - q0 b and q = RN(q0 + r inv), q is
RN(s / b) for every FP64 s and integer 1 <= b < 2^31."""
import math
import random
from fractions import Fraction as F


def _fma(a, b, c):
    return float(F(a) * F(b) + F(c))     # float of a Fraction rounds to nearest even


def _div_by(s, b):
    inv = 1.0 / b
    q0 = s * inv
    r = _fma(-q0, float(b), s)
    assert F(r) == F(s) - F(q0) * b      # the residual is exact
    return _fma(r, inv, q0)


def test_quotient_equals_division():
    rng = random.Random(11)
    for _ in range(40000):
        b = rng.choice([rng.randint(1, 300), rng.randint(1, 2**31 - 1), 2**rng.randint(0, 30) + rng.randint(-1, 1) or 1])
        b = max(1, min(b, 2**31 - 1))
        s = math.ldexp(rng.uniform(-1, 1), rng.randint(-300, 300))
        if rng.random() < 0.3:           # quotients next to a rounding boundary
            q = math.ldexp(1.0 + rng.getrandbits(52) * 2.0**-52, rng.randint(-40, 40))
            s = math.nextafter(float((F(q) + F(math.ulp(q)) / 2) * b), rng.choice([-math.inf, math.inf]))
        assert _div_by(s, b) == s / b, (s, b)
