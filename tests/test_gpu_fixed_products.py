"""GPU: products of lines of doubles with an operator on the integer pipes (fx_apply of
csrc/fixed.cuh), called by themselves through tests/fixed_probe.cu, against exact rational
arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from oracle.basis import Basis
from paper_1406_7416_gb300 import build_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("probe") / "fixed_probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fixed_probe.cu")
    subprocess.run([build_lib._nvcc()] + build_lib.NVCC_FLAGS + ["-shared", src, "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def products(probe):
    ptr = np.ctypeslib.ndpointer(np.float64, flags="C")
    probe.fixed_products.argtypes = [ctypes.c_int, ptr, ptr, ctypes.c_longlong, ptr]

    def call(M, x):
        M, x = np.ascontiguousarray(M, float), np.ascontiguousarray(x, float)
        out = np.empty_like(x)
        assert probe.fixed_products(M.shape[0], M, x, x.shape[0], out) == 0
        return out
    return call


def _exact(M, x):
    """The exact products as Fractions."""
    F = [[Fraction(float(v)) for v in row] for row in M]
    return [[sum(m * Fraction(float(v)) for m, v in zip(row, line)) for row in F] for line in x]


def _lines(n, count, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(-1, 1, (count, n)) * 2.0 ** rng.integers(-4, 1, (count, n)) * \
        2.0 ** rng.integers(-60, 60, (count, 1))


@pytest.mark.parametrize("n", range(2, 11))
def test_cancelling_products_are_zero(products, n):
    """An antisymmetric row on a line of equal elements, and rows of a line of zeros, give zero."""
    rng = np.random.default_rng(n)
    half = rng.uniform(0.1, 3.0, (n, n // 2))
    mid = np.zeros((n, n % 2))
    M = np.concatenate([half, mid, -half[:, ::-1]], axis=1)
    x = np.repeat(_lines(1, 500, n), n, axis=1)
    x[::7] = 0.0
    x[1::7] = 3.0
    x[2::7] = -0.25
    assert np.array_equal(products(M, x), np.zeros_like(x))


@pytest.mark.parametrize("n", range(1, 11))
def test_products_are_odd(products, n):
    """f(-x) = -f(x), bit for bit, small whole numbers (whose products end in zero bits) included."""
    rng = np.random.default_rng(n)
    M = rng.uniform(-2, 2, (n, n))
    x = _lines(n, 2000, 3 * n)
    x[::3] = rng.integers(-4, 5, x[::3].shape)
    y = products(M, x)
    assert np.array_equal(products(M, -x), -y)
    assert np.abs(y).max() > 0


@pytest.mark.parametrize("n", range(1, 11))
def test_products_against_exact_ones(products, n):
    """Error of each output in units of s m, s the operator's largest row sum and m the line's
    largest magnitude: elements cut at 2^-58 m, entries rounded at 2^-62 s, the n products of low
    halves left out (each below 2^-57), the sum cut at 2^-55, and the result rounded to 53 bits."""
    M = Basis(n - 1).D if n > 1 else np.array([[1.7]])
    x = _lines(n, 150, 7 * n)
    y = products(M, x)
    s, m = np.abs(M).sum(axis=1).max(), np.abs(x).max(axis=1)
    bar = Fraction(1, 2 ** 58) + n * Fraction(1, 2 ** 62) + n * Fraction(1, 2 ** 57) + \
        Fraction(1, 2 ** 55) + Fraction(1, 2 ** 53)
    worst = 0.0
    for l, row in enumerate(_exact(M, x)):
        for a, v in enumerate(row):
            err = abs(Fraction(float(y[l, a])) - v)
            assert err <= bar * Fraction(float(s)) * Fraction(float(m[l])), (l, a, float(err))
            worst = max(worst, float(err) / (s * m[l]))
    print(n, worst)


@pytest.mark.parametrize("n", [1, 2, 3, 6, 9, 10])
@pytest.mark.parametrize("e", [-1060, -1000, -962, -958, 974, 980, 1010])
def test_lines_at_the_ends_of_the_range(products, n, e):
    """Lines below 2^-959 (subnormals too) and from 2^977 on: every product rounds at 2^-53 of
    its terms, or at the last place of a subnormal."""
    M = Basis(n - 1).D if n > 1 else np.array([[1.7]])
    x = np.ldexp(_lines(n, 40, n), 0)
    x = np.ldexp(x / np.abs(x).max(axis=1, keepdims=True), e)
    x[3] = 0.0
    y = products(M, x)
    s, m = np.abs(M).sum(axis=1).max(), np.abs(x).max(axis=1)
    for l, row in enumerate(_exact(M, x)):
        for a, v in enumerate(row):
            bar = (n + 1) * Fraction(float(s)) * Fraction(float(m[l])) / 2 ** 53 + n * Fraction(1, 2 ** 1074)
            assert abs(Fraction(float(y[l, a])) - v) <= bar, (l, a)


@pytest.mark.parametrize("n", range(1, 11))
@pytest.mark.parametrize("e", [-1060, -1000, -958, 0, 974, 980, 1010])
def test_row_sums_over_the_range(probe, n, e):
    """The first time solve, each row's sum times one value: an operator entry and the result round."""
    M = Basis(n - 1).Ktau if n > 1 else np.array([[1.7]])
    rng = np.random.default_rng(n)
    x = np.repeat(np.ldexp(rng.uniform(0.5, 1, (30, 1)) * rng.choice([-1, 1], (30, 1)), e), n, axis=1)
    x[3] = 0.0
    y = np.empty_like(x)
    ptr = np.ctypeslib.ndpointer(np.float64, flags="C")
    probe.fixed_sums.argtypes = [ctypes.c_int, ptr, ptr, ctypes.c_longlong, ptr]
    assert probe.fixed_sums(n, np.ascontiguousarray(M), x, x.shape[0], y) == 0
    sums = [sum(Fraction(float(v)) for v in row) for row in M]
    scale = Fraction(float(np.abs(M).sum(axis=1).max()))
    for l in range(x.shape[0]):
        for a in range(n):
            v = sums[a] * Fraction(float(x[l, a]))
            # the row's sum in doubles (n roundings), the product, and in integers 2^-55 of the scale
            bar = (n + 4) * scale * abs(Fraction(float(x[l, a]))) / 2 ** 53 + Fraction(1, 2 ** 1074)
            assert abs(Fraction(float(y[l, a])) - v) <= bar, (l, a)


@pytest.mark.parametrize("n", [1, 2, 5])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_lines_with_a_nan_or_an_infinity(products, n, bad):
    x = np.ones((6, n))
    x[2, n // 2] = bad
    y = products(np.full((n, n), 1.5), x)
    assert not np.isfinite(y[2]).any() and np.isfinite(np.delete(y, 2, axis=0)).all()


def _operators(n):
    from oracle.subcell import projection_matrix
    b = Basis(n - 1)
    P = projection_matrix(b, 2 * n - 1)
    ops = {"D": b.D, "Mvol": b.w[None, :] * b.D.T / b.w[:, None]}
    if n > 2:                               # (P of two nodes is not formed by these products)
        ops.update(P_low=P[:n], P_mid=P[n // 2:n // 2 + n])
    return ops


@pytest.mark.parametrize("k", [7, 20, 40])
@pytest.mark.parametrize("n", range(2, 11))
def test_steep_lines(products, n, k):
    """Lines with a spike at each node, and with a jump between each two, of 2^k: every row is as
    accurate as an FMA chain, whose n roundings are each below 2^-53 of the sum of the terms'
    magnitudes, a row that gives the large side little or no weight among them."""
    rng = np.random.default_rng(n + k)
    shapes = [np.arange(n) == j for j in range(n)] + [np.arange(n) < j for j in range(1, n)] + \
        [np.arange(n) >= j for j in range(1, n)]
    x = np.array([np.where(s, 2.0 ** k, 1.0) for s in shapes] * 4)
    x *= rng.uniform(1, 1.9, x.shape) * rng.choice([-1, 1], x.shape)
    for name, M in _operators(n).items():
        y = products(M, x)
        for l, row in enumerate(_exact(M, x)):
            for a, v in enumerate(row):
                mags = sum(abs(Fraction(float(m)) * Fraction(float(t))) for m, t in zip(M[a], x[l]))
                err = abs(Fraction(float(y[l, a])) - v)
                assert err <= n * mags / 2 ** 53, (name, l, a, float(err / mags) * 2 ** 53)


def test_widened_floats_are_exact(probe):
    """FP32 results of the predictor's sweeps that an FP64 sweep goes on from: every float as its
    double, subnormal ones, signed zeros and infinities included."""
    rng = np.random.default_rng(1)
    bits = np.concatenate([rng.integers(0, 2 ** 32, 20000), rng.integers(0, 2 ** 23, 2000),
                           2 ** 31 + rng.integers(0, 2 ** 23, 2000),
                           [0, 1, 2 ** 31, 2 ** 31 + 1, 2 ** 23 - 1, 2 ** 23, 0x7f800000, 0xff800000]])
    x = bits.astype(np.uint32).view(np.float32)
    x = x[~np.isnan(x)]
    out = np.empty(x.size)
    assert probe.widen_floats(x.ctypes.data_as(ctypes.c_void_p), x.size, out.ctypes.data_as(ctypes.c_void_p)) == 0
    np.testing.assert_array_equal(out.view(np.uint64), x.astype(np.float64).view(np.uint64))
