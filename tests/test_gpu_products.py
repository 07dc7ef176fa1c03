"""The FP64 triple products element by element against exact integer arithmetic.

Both kernels read a block (or tile of 32 x 32) as integers under one exponent, so their error is
bounded relative to the largest elements and not element by element.  The bounds below follow
from what is rounded or left out, with M = the largest |element| of an operand, u = 2^-53:

prepared operands (58 bits; products by digits of 10 bits, depths of 16 at a time)
  X, Y, Z              2^-58 M each
  T = X Y              n 2^-57 Mx My, and per depth of 16 two units of 2^-54 Mx My: the rounding
                       of the low orders' FP32 sum and the orders that are left out
  T to 58 bits         2^-58 Mt (exact where T is small)
  T Z                  p 2^-57 Mt Mz, and per depth of 16 two units of 2^-54 Mt Mz
general kernel (57 bits in limbs of 29; depths of 32)
  X, Y, Z              2^-57 M each, and lo lo' <= 2^-56 Mx My left out: n 2^-55 Mx My
  T                    per chunk of 32 one unit of 2^(extra - 54) Mx My, extra = bits for n / 32 sums
  T to 57 bits, T Z    p 2^-55 Mt Mz and 2^-54 Mt Mz per chunk
and the FP64 sum over the tasks.
"""
import math

import numpy as np
import pytest

from paper_2001_04890_gb300 import binding

pytestmark = pytest.mark.gpu

SHIFT = 300


def _int(x):
    """x 2^SHIFT as Python integers, exactly."""
    def one(v):
        m, e = math.frexp(float(v))
        k = e - 53 + SHIFT
        i = int(m * 2.0**53)
        assert k >= 0
        return i << k
    return np.array([[one(v) for v in row] for row in x], dtype=object)


def _exact(X, Y, Z, f):
    """sum_t f_t X_t Y Z_t as integers in units of 2^(-4 SHIFT)."""
    y = _int(Y)
    out = 0
    for t in range(len(f)):
        d = _int(X[t]) @ y @ _int(Z[t])
        out = out + d * _int([[f[t]]])[0, 0]
    return out


def _bound(X, Y, Z, f, prepared):
    n, p = Y.shape
    total, sums = 0.0, 0.0
    for t in range(len(f)):
        mx, my, mz = np.abs(X[t]).max(), np.abs(Y).max(), np.abs(Z[t]).max()
        mt = max(np.abs(X[t] @ Y).max(), 2.0**-22 * mx * my)
        if prepared:
            dt = (n * 2.0**-57 + math.ceil(n / 16) * 2.0**-53) * mx * my
            d = p * (dt * mz + 2.0**-57 * mt * mz + 2.0**-58 * mt * mz) + math.ceil(p / 16) * 2.0**-53 * mt * mz
        else:
            chunks = math.ceil(n / 32)
            dt = (n * 2.0**-55 + chunks * 2.0**(math.ceil(math.log2(chunks)) + (chunks > 1) - 54)) * mx * my
            d = p * (dt + 2.0**-55 * mt + 2.0**-57 * mt) * mz + math.ceil(p / 32) * 2.0**-54 * mt * mz
        total += abs(f[t]) * d
        sums += abs(f[t]) * (np.abs(X[t] @ Y) @ np.abs(Z[t])).max()
    return total + 2.0**-53 * (len(f) * math.ceil(p / 16) + 4) * sums


def _error(D, exact):
    """|D - exact| as floats."""
    d = _int(D) * (1 << (3 * SHIFT)) - exact
    return np.array([[float(abs(int(v)) >> 200) * 2.0**(200 - 4 * SHIFT) for v in row] for row in d])


SHAPES = [(5, 7, 6, 9), (16, 16, 16, 16), (17, 30, 20, 33), (33, 40, 48, 64), (70, 100, 24, 100)]


@pytest.mark.parametrize("prepared", [True, False])
@pytest.mark.parametrize("m,n,p,q", SHAPES)
@pytest.mark.parametrize("grade", [0, 1, 3])
def test_graded_inside_a_block(grade, m, n, p, q, prepared):
    """Rows and columns that fall off by 2^-grade each: the error is bounded by the largest elements
    of the blocks, for the small elements of D too."""
    rng = np.random.default_rng(7)
    fall = lambda k: np.ldexp(1.0, -grade * (np.arange(k) % 24))  # noqa: E731
    X = rng.standard_normal((3, m, n)) * fall(m)[:, None]
    Y = rng.standard_normal((n, p)) * fall(n)[:, None] * fall(p)
    Z = rng.standard_normal((3, p, q)) * fall(q)
    f = [1.0, -0.7, 0.3]
    D = binding.selftest_chain(X, Y, Z, f, prepared=prepared)
    err = _error(D, _exact(X, Y, Z, f))
    assert err.max() <= _bound(X, Y, Z, f, prepared)


def _digits(rng, n, top):
    """n integers whose five lower digits are at -512..-500 (the last -512: the value has 53 bits)."""
    d = rng.integers(-512, -499, (n, 6))
    d[:, 0], d[:, 5] = top, -512
    return [sum(int(x) << (10 * (5 - i)) for i, x in enumerate(row)) for row in d]


@pytest.mark.parametrize("depth", [16, 8])
@pytest.mark.parametrize("m,p", [(5, 7), (16, 16), (33, 40), (70, 100)])
def test_no_digit_order_is_missing(m, p, depth):
    """Largest digits of one sign in the last chunk of a dot product, whose sum the first chunk cancels to the
    last bits.  The FP32 sums G_5 and G_6 pass 2^24 here.  Two units of 2^60 are allowed (the
    low orders' rounding in either chunk is 1.1 and 0.7 units, orders above 6 are 2^-6); without
    order 6 the result is off by 19.8 of them (depth 8: 9.9)."""
    rng = np.random.default_rng(11)
    a, b = _digits(rng, depth, -250), _digits(rng, depth, -250)
    S = sum(x * y for x, y in zip(a, b))
    u = 255 << 50
    w = -(S // (16 * u) >> 5 << 5)
    R = S + 16 * u * w
    assert abs(R) < 1 << 68 and abs(w) < 1 << 58
    x = np.array([u] * 16 + a, dtype=object)
    y = np.array([w] * 16 + b, dtype=object)
    xf, yf = (np.array([math.ldexp(int(v), -57) for v in z]) for z in (x, y))
    assert all(int(math.ldexp(float(g), 57)) == v for z, h in ((x, xf), (y, yf)) for v, g in zip(z, h))
    D = binding.selftest_chain(np.broadcast_to(xf, (1, m, 16 + depth)), np.repeat(yf[:, None], p, 1), None, [1.0])
    got = np.ldexp(D, 54)  # in units of 2^60
    assert np.max(np.abs(got - R / 2.0**60)) <= 2.0


@pytest.mark.parametrize("n", [31, 32, 33, 119, 120])
def test_largest_values_at_the_longest_inner_dimension(n):
    """Every element just below 2: the 64-bit sums come closest to their limit at n = 120."""
    big = 2.0 - 2.0**-52
    X, Y, Z = np.full((2, 9, n), big), np.full((n, 18), big), np.full((2, 18, 35), -big)
    for prepared in (True, False):
        for sign in (1.0, -1.0):
            D = binding.selftest_chain(sign * X, Y, Z, [1.0, 1.0], prepared=prepared)
            assert _error(D, _exact(sign * X, Y, Z, [1.0, 1.0])).max() <= _bound(X, Y, Z, [1.0, 1.0], prepared)


def test_longer_inner_dimensions_are_refused_by_the_prepared_kernels_only():
    rng = np.random.default_rng(13)
    X, Y, Z = rng.standard_normal((1, 20, 121)), rng.standard_normal((121, 10)), rng.standard_normal((1, 10, 20))
    with pytest.raises(binding.DMRGError) as err:
        binding.selftest_chain(X, Y, Z, [1.0])
    assert err.value.code == binding.DMRG_EINVAL
    D = binding.selftest_chain(X, Y, Z, [1.0], prepared=False)
    assert _error(D, _exact(X, Y, Z, [1.0])).max() <= _bound(X, Y, Z, [1.0], False)


@pytest.mark.parametrize("prepared", [True, False])
@pytest.mark.parametrize("m,n,p,q", SHAPES)
def test_fp32_operators(m, n, p, q, prepared):
    """FP32 products: each of the n + p multiply-adds and the three roundings by 2^-24."""
    rng = np.random.default_rng(17)
    X, Y, Z, f = (rng.standard_normal(s) for s in ((3, m, n), (n, p), (3, p, q), 3))
    D = binding.selftest_chain(X, Y, Z, f, fp32=True, prepared=prepared)
    ref = sum(f[t] * (X[t] @ Y @ Z[t]) for t in range(3))
    big = sum(abs(f[t]) * (np.abs(X[t]) @ np.abs(Y) @ np.abs(Z[t])) for t in range(3))
    assert np.all(np.abs(D - ref) <= 2.0**-24 * (n + p + 8) * big)
