"""CPU model of the quotients and square roots that the FP64 kernels take from a shared reciprocal with
one residual correction: bit for bit the rounded quotient and root, over random significands, the
quotients closest to a rounding boundary, zeros, and the exponents where the residual is no longer
exact (there the division itself decides)."""
import ctypes
import math
import random

import pytest

libm = ctypes.CDLL("libm.so.6")
libm.fma.restype = ctypes.c_double
libm.fma.argtypes = [ctypes.c_double] * 3
fma = libm.fma


def _divide(n, d):
    if d == 0.0 or math.isnan(n) or math.isnan(d):
        return math.nan if n == 0.0 or math.isnan(n) or math.isnan(d) else math.copysign(
            math.inf, n) * math.copysign(1.0, d)
    return n / d


def _quotient(n, d, r, calls):
    """quotient() of lw_deposit.cu."""
    q0 = n * r
    if n == 0.0 and q0 == 0.0:
        return q0
    q = fma(fma(-q0, d, n), r, q0)
    if not (2.0 ** -960 <= abs(n) and 2.0 ** -960 <= abs(q) < math.inf):
        calls.append(1)
        return _divide(n, d)
    return q


def _same(a, b):
    return a == b and math.copysign(1.0, a) == math.copysign(1.0, b) or (a != a and b != b)


def _significands(rng, count):
    for _ in range(count):
        yield 1.0 + rng.getrandbits(52) * 2.0 ** -52, 1.0 + rng.getrandbits(52) * 2.0 ** -52


def test_quotients():
    rng, calls = random.Random(3), []
    for n, d in _significands(rng, 100000):
        n = math.ldexp(n, rng.randint(-300, 100)) * rng.choice((-1.0, 1.0))
        d = math.ldexp(d, rng.randint(-120, 3))
        assert _same(_quotient(n, d, 1.0 / d, calls), n / d)
    assert not calls


@pytest.mark.parametrize("shift", [53, 54])
def test_quotients_next_to_a_rounding_boundary(shift):
    """2^shift n = (2 h + 1) d +- k: n/d within k 2^-54 ulp or so of the middle of two doubles."""
    rng, tried = random.Random(shift), 0
    for _ in range(20000):
        d = (1 << 53) - 1 - 2 * rng.randrange(1 << rng.randint(1, 51))
        inverse = pow(1 << shift, -1, d)
        for k in (-5, -3, -1, 1, 3, 5):
            n = k * inverse % d
            if shift == 53:   # quotients in [1, 2)
                n += d
            if 1 << 52 <= n < 1 << 53:
                tried += 1
                assert _same(_quotient(float(n), float(d), 1.0 / d, []), n / d)
    assert tried > 1000


@pytest.mark.parametrize("exponent", [-1074, -1060, -1022, -1000, -970, -961, -960, 900, 1000, 1023])
def test_quotients_at_the_ends_of_the_range(exponent):
    rng, calls = random.Random(exponent), []
    for n, d in _significands(rng, 5000):
        n = math.ldexp(n, exponent)
        d = math.ldexp(d, rng.choice((-160, -60, -1, 0, 3, 40)))
        assert _same(_quotient(n, d, _divide(1.0, d), calls), _divide_safe(n, d))


def _divide_safe(n, d):
    try:
        return n / d
    except OverflowError:
        return math.copysign(math.inf, n)


@pytest.mark.parametrize("n", [0.0, -0.0, 1.5, math.inf, math.nan])
@pytest.mark.parametrize("d", [0.0, 5e-324, 1e-310, 1.5, math.inf, math.nan])
def test_quotients_of_special_values(n, d):
    r = _divide(1.0, d)
    assert _same(_quotient(n, d, r, []), _divide(n, d))


def test_square_roots():
    """root() of lw_push.cu, from a reciprocal root that is off by up to an ulp either way."""
    rng = random.Random(5)
    for m, _ in _significands(rng, 60000):
        a = math.ldexp(m, rng.randint(0, 60))
        if rng.random() < 0.5:   # next to a square of a middle of two doubles
            h = (1 << 52) + rng.getrandbits(52)
            a = float((2 * h + 1) ** 2 >> rng.choice((53, 54))) * 2.0 ** -50
        y0 = 1.0 / math.sqrt(a)
        for y in (math.nextafter(y0, 0.0), y0, math.nextafter(y0, 2.0)):
            g = a * y
            assert fma(fma(-g, g, a), 0.5 * y, g) == math.sqrt(a)
