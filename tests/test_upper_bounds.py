"""Host checks of the upper bounds (FP32 mantissa, integer exponent) that choose the
exponents of the fixed-point vectors and so keep their int64 entries from
overflowing (scalar_bounds.cuh compiled for the host): against exact fractions, at
carries (mantissas next to 2), exponent differences around the 40 bits that an
addition keeps, zeros, subnormals, the ends of the exponent range and int64 limits.

Each operation rounds up and may lose 2^-22 (its factor) plus two FP32 roundings of
2^-24 at most; the conversions lose one unit of a 23-bit mantissa."""

import random
from fractions import Fraction

import numpy as np
import pytest

from paper_1102_5071_gb300 import _capi
from paper_1102_5071_gb300.build import build


@pytest.fixture(scope="module")
def lib():
    build()
    return _capi.load()


def _bounds(lib, op, a=None, b=None, v=None):
    n = len(v if op == 1 else a)
    arr = [np.array(x, dtype=t) if x is not None else None for x, t in ((a, np.float64), (b, np.float64), (v, np.int64))]
    m, e, e57 = np.zeros(n, dtype=np.float32), np.zeros(n, dtype=np.int32), np.zeros(n, dtype=np.int32)
    ptr = [x.ctypes.data if x is not None else None for x in arr]
    assert lib.cfet_selftest_upper_bounds(op, *ptr, n, m.ctypes.data, e.ctypes.data, e57.ctypes.data) == _capi.CFET_OK
    out = []
    for i in range(n):
        assert m[i] == 0.0 or 1.0 <= m[i] <= 2.0
        val = Fraction(float(m[i])) * Fraction(2) ** int(e[i])
        # the exponent: val < 2^(57 + E), and no smaller one would do
        if val == 0 or not Fraction(2) ** -963 <= val < Fraction(2) ** 964:
            assert e57[i] == -960
        else:
            assert val < Fraction(2) ** (57 + int(e57[i])) <= 2 * val
        out.append(val)
    return out


def _doubles(rng, n, emax=900):
    near = [1.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1), 2.0 - 2.0 ** -23, 2.0 - 2.0 ** -24, 2.0 - 2.0 ** -25,
            1.0 + 2.0 ** -23, 1.5, 1.0 + 2.0 ** -24]
    out = []
    for _ in range(n):
        m = rng.choice(near) if rng.random() < 0.5 else 1.0 + rng.random()
        out.append((1 if rng.random() < 0.5 else -1) * float(np.ldexp(m, rng.randint(-emax, emax))))
    return out


def test_conversions_never_round_down(lib):
    rng = random.Random(11)
    a = _doubles(rng, 600, 1000) + [0.0, -0.0, 2.0 ** -1022, np.finfo(float).max, -np.finfo(float).max]
    for x, u in zip(a, _bounds(lib, 0, a)):
        x = abs(Fraction(x))
        assert x <= u <= x * (1 + Fraction(1, 1 << 22))
    sub = [5e-324, -1e-310, float(np.nextafter(2.0 ** -1022, 0))]
    assert all(u == Fraction(2) ** -1022 for u in _bounds(lib, 0, sub))
    v = [-1, 0, 1, 2, 3, (1 << 24) - 1, (1 << 24) + 1, (1 << 25) - 1, (1 << 57) - 1, 1 << 57, (1 << 60) + 1, (1 << 62) - 1,
         1 << 62, (1 << 63) - 1] + [rng.getrandbits(b) for b in range(1, 64) for _ in range(8)]
    for x, u in zip(v, _bounds(lib, 1, v=v)):
        x = Fraction(max(x, 0))
        assert x <= u <= x * (1 + Fraction(1, 1 << 22))


def test_products_and_sums_never_round_down(lib):
    rng = random.Random(12)
    loss = Fraction(1, 1 << 21)  # 2^-22 and the roundings, and those of the two operands below
    conv = Fraction(1, 1 << 22)
    a, b = _doubles(rng, 1500, 400), _doubles(rng, 1500, 400)
    # additions: exponents 0 to 60 apart, around the 40 bits kept
    for d in range(-60, 61):
        a.append(float(np.ldexp(rng.choice([1.0, 2.0 - 2.0 ** -24, 1.0 + rng.random()]), d)))
        b.append(rng.choice([1.0, -(2.0 - 2.0 ** -24), 1.0 + rng.random()]))
    a += [0.0, 0.0, 3.0, 2.0 - 2.0 ** -52, 2.0 ** -1022, 0.0]
    b += [0.0, 5.0, 0.0, 2.0 - 2.0 ** -52, 2.0 ** -1022, 2.0 - 2.0 ** -52]
    for op in (2, 3):
        for x, y, u in zip(a, b, _bounds(lib, op, a, b)):
            x, y = abs(Fraction(x)), abs(Fraction(y))
            ref = x * y if op == 2 else x + y
            assert ref <= u <= ref * (1 + loss) * (1 + conv) ** 2, (op, float(x), float(y))


def test_norm_shift(lib):
    rng = random.Random(13)
    v = [0, -3, 1, 2, 3, (1 << 61) - 1, 1 << 61, (1 << 62) - 1, 1 << 62, (1 << 63) - 1]
    v += [rng.getrandbits(b) for b in range(1, 64) for _ in range(8)]
    v += [30 * m for m in ((1 << 57) - 1, 1 << 57)]  # neighbour sums of the longest chain
    arr, out = np.array(v, dtype=np.int64), np.zeros(len(v), dtype=np.int32)
    assert lib.cfet_selftest_norm_shift(arr.ctypes.data, len(v), out.ctypes.data) == _capi.CFET_OK
    for x, s in zip(v, out):
        if x <= 0 or x >= 1 << 62:
            assert s == 0
        else:
            assert 1 << 61 <= x << int(s) < 1 << 62
    assert all(30 * m < 1 << 62 for m in ((1 << 57) - 1, 1 << 57))
