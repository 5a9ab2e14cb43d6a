"""Host model of the exact slicing of FP64 into bf16 digits that the FP64 tensor-core kernels share (csrc/oz.cuh):
62 fractional bits below the vector's exponent, eight balanced base-256 digits, the 36 digit products p + q <= 7
summed exactly over at most 128 entries, and the two 64-bit sums hi and lo.  Checked with Python integers: the digits
reconstruct the rounded entry and are exact in bf16, every FP32 accumulator stays an exact integer, and the product
lies within K 2^-60 2^(e_x + e_y) of the exact sum (rounding to 62 bits costs 2^-63 of the largest entry in each
factor, the dropped pairs at most 8 K 2^14 2^-76 of it, both well inside)."""
from fractions import Fraction

import numpy as np
import pytest


def exponent(x):
    """|x_k| < 2^e, from the largest high word as the kernels take it."""
    be = int(np.max(np.abs(x)).view(np.uint64) >> np.uint64(52))
    return max(be - 1022, -900)


def cut(x, e):
    """The eight signed digits of x, most significant first."""
    if x == 0 or abs(x) < 2.0 ** -1022:
        return [0] * 8
    v = Fraction(float(x)) * Fraction(2) ** (62 - e)
    mag = (abs(v) + Fraction(1, 2)).__floor__()  # half away from zero
    I = -mag if x < 0 else mag
    assert abs(I) <= 2 ** 62
    out = []
    for _ in range(7):
        d = (I + 128) % 256 - 128
        out.append(d)
        I = (I - d) // 256
    out.append(I)
    return out[::-1]


@pytest.mark.parametrize("seed", range(6))
def test_digits_and_product(seed):
    rng = np.random.default_rng(seed)
    for K in (1, 31, 32, 128):
        spread = int(rng.integers(0, 40))
        x, y = (rng.normal(size=K) * np.exp2(-rng.integers(0, spread + 1, size=K)) for _ in range(2))
        if seed == 0:  # the worst case of the accumulators: every entry at the top of its range
            x = y = np.full(K, -(2.0 - 2.0 ** -52))
        ex, ey = exponent(x), exponent(y)
        dx, dy = np.array([cut(v, ex) for v in x], dtype=object), np.array([cut(v, ey) for v in y], dtype=object)
        for v, d in zip(x, dx):
            assert all(-128 <= t <= 127 for t in d[1:]) and abs(d[0]) <= 64
            back = sum(Fraction(int(t)) * Fraction(256) ** (7 - p) for p, t in enumerate(d)) * Fraction(2) ** (ex - 62)
            assert abs(back - Fraction(float(v))) <= Fraction(2) ** (ex - 63)
        acc = []
        for d in range(8):
            terms = [int(a) * int(b) for p in range(d + 1) for a, b in zip(dx[:, p], dy[:, d - p])]
            assert sum(abs(t) for t in terms) <= 2 ** 24  # every partial sum is exact in FP32
            acc.append(sum(terms))
        hi = sum(a * 256 ** (3 - d) for d, a in enumerate(acc[:4]))
        lo = sum(a * 256 ** (7 - d) for d, a in enumerate(acc) if d >= 4)
        assert abs(hi) < 2 ** 45 and abs(lo) < 2 ** 50
        got = (hi * 2 ** 32 + lo) * Fraction(2) ** (ex + ey - 68)
        exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(x, y))
        assert abs(got - exact) <= K * Fraction(2) ** (ex + ey - 60)
