"""Host models of the digit products' error bound (csrc/oz.cuh) at its worst case, and of the apply's own cut
(csrc/kern_apply_oz.cu), with Python integers."""
from fractions import Fraction

import numpy as np
import pytest

from test_digit_model import cut, exponent


def product(x, y):
    """(value of the kernels' sum, exact sum) in units of 2^(e_x + e_y)."""
    ex, ey = exponent(x), exponent(y)
    dx, dy = [cut(v, ex) for v in x], [cut(v, ey) for v in y]
    got = sum(a[p] * b[q] * 256 ** (14 - p - q) for a, b in zip(dx, dy) for p in range(8) for q in range(8 - p))
    exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(x, y))
    return Fraction(got, 2 ** 124), exact / Fraction(2) ** (ex + ey)


@pytest.mark.parametrize("K", [1, 2, 32, 128])
def test_dropped_pairs_worst_case(K):
    """Every dropped pair at its largest (digits of -128 after a large first entry): the error passes K 2^-60, and stays
    below what the seven pairs p + q = 8 (2^14 2^48 2^-124 each), the fewer ones beyond and the two roundings allow."""
    x = np.full(K, -float.fromhex("0x1.0101010101010p-7"))
    if K > 1:
        x[0] = 0.75
    got, exact = product(x, x)
    bound = K * (sum(Fraction(15 - s, 1) * Fraction(2) ** (14 + 8 * (14 - s) - 124) for s in range(8, 15)) + Fraction(1, 2 ** 62))
    assert bound < K * Fraction(2) ** -58
    assert abs(got - exact) <= bound
    if K >= 32:
        assert abs(got - exact) > K * Fraction(2) ** -60


def dig_bytes(x, e):
    """The apply's cut: bytes (digit + 128) of x truncated to 62 fractional bits below 2^e, most significant first."""
    bits = int(np.float64(x).view(np.uint64))
    be, man, neg = bits >> 52 & 0x7FF, bits & (1 << 52) - 1, bits >> 63
    M = (man | 1 << 52) << 10
    n = min(1023 + e - be, 63)
    assert n >= 1
    I = -(M >> n) if neg else M >> n
    return [(I + 0x8080808080808080) % 2 ** 64 >> 56 - 8 * p & 0xFF for p in range(8)]


@pytest.mark.parametrize("seed", range(5))
def test_apply_cut(seed):
    """The bytes are the digits plus 128, the digits give x truncated at 2^(e - 62) (zeros give zero digits), and the row
    sums of 64 products with all 64 digit pairs, put together as the kernel does, are exact in its integer types."""
    rng = np.random.default_rng(seed)
    x, y = (rng.normal(size=64) * np.exp2(-rng.integers(0, 45, size=64)) for _ in range(2))
    if seed == 0:
        x = y = np.full(64, -(2.0 - 2.0 ** -52))
    if seed == 1:
        x[1:], y[1:] = -float.fromhex("0x1.0101010101010p-7"), -float.fromhex("0x1.0101010101010p-7")
        x[0] = y[0] = 0.75
    x[-1] = 0.0
    ex, ey = exponent(x), exponent(y)
    dx, dy = [[b - 128 for b in dig_bytes(v, ex)] for v in x], [[b - 128 for b in dig_bytes(v, ey)] for v in y]
    assert dx[-1] == [0] * 8
    val = lambda d, e: sum(t * 256 ** (7 - p) for p, t in enumerate(d)) * Fraction(2) ** (e - 62)  # noqa: E731
    for v, d, e in [(v, d, ex) for v, d in zip(x, dx)] + [(v, d, ey) for v, d in zip(y, dy)]:
        assert abs(val(d, e) - Fraction(float(v))) < Fraction(2) ** (e - 62) and abs(val(d, e)) <= abs(float(v))
    acc = [[sum(a[p] * b[q] for a, b in zip(dx, dy)) for q in range(8)] for p in range(8)]
    assert all(abs(t) <= 2 ** 24 for r in acc for t in r)  # exact in FP32
    total = Fraction(0)
    for t in range(4):  # lane t holds the digits q = 2 t and 2 t + 1 of the vector
        u = [(acc[j][2 * t] if j < 8 else 0) + (acc[j - 1][2 * t + 1] if j > 0 else 0) for j in range(9)]
        assert all(abs(u[j] * 256 + u[j + 1]) < 2 ** 31 for j in (0, 2, 5, 7))
        hi = ((u[0] * 256 + u[1]) * 65536 + (u[2] * 256 + u[3])) * 256 + u[4]
        lo = (u[5] * 256 + u[6]) * 65536 + (u[7] * 256 + u[8])
        assert abs(hi) < 2 ** 63 and abs(lo) < 2 ** 63
        total += (hi * 2 ** 32 + lo) * Fraction(2) ** (ex + ey - 76 - 16 * t)
    assert total == sum(val(a, ex) * val(b, ey) for a, b in zip(dx, dy))
