"""The FP64 contraction in digit form (exact BF16 digit products, csrc/gemm_f64e.cu) against exact
rational arithmetic, at the edges of its tiles, chunks and K ranges.

Bound.  Each operand is rounded to 62 bits of its row's power of two 2^E (at most twice the row's
largest element), and the digit pairs beyond level 7 are dropped: 7 pairs of at most 2^14 with the
weight 2^-76, i.e. 7 2^-62 2^(EA+EB) <= 2^-57 max|a| max|b| per k, the operands' rounding included.
One final rounding gives 2^-53 |c|; twice that is allowed for coherent sums, whose levels 5 to 7 may
round in FP32, and for the sum over K ranges."""
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def contraction(A, B):
    need_gpu()
    from paper_1703_01545_gb300 import _lib
    lib = _lib.load()
    Md, Nd, K = A.shape[0], B.shape[0], A.shape[1]
    C = np.empty((Nd, Md))
    code = lib.afqmc_test_gemm(0, Md, Nd, K, A.ctypes.data, B.ctypes.data, 1.0, C.ctypes.data, None)
    assert code == 0
    return C


def check(A, B, C, rng, samples=300):
    Md, Nd, K = A.shape[0], B.shape[0], A.shape[1]
    m = np.concatenate([[0, Md - 1, 0, Md - 1], rng.integers(0, Md, samples)])
    n = np.concatenate([[0, Nd - 1, Nd - 1, 0], rng.integers(0, Nd, samples)])
    for i, j in zip(m, n):
        exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(A[i], B[j]))
        bound = 2.0 ** -52 * abs(float(exact)) + K * 2.0 ** -57 * np.abs(A[i]).max() * np.abs(B[j]).max()
        assert abs(float(Fraction(float(C[j, i])) - exact)) <= bound + 1e-320, (i, j)


# (Md, Nd, K): tile edges in both roles (rows in 128, columns in 64), one and several chunks of 256 k,
# K padding, split K ranges (few tiles, long K), several chunks of B rows
SHAPES = [(128, 4096, 64), (129, 4031, 65), (2080, 193, 320), (64, 8191, 64), (1, 4096, 8192),
          (480, 256, 2305), (65, 1500, 511), (300, 700, 256), (300, 700, 257), (33, 30000, 32)]


@pytest.mark.parametrize("Md,Nd,K", SHAPES)
def test_against_exact_arithmetic(Md, Nd, K):
    rng = np.random.default_rng(Md * 7 + Nd * 3 + K)
    A = rng.standard_normal((Md, K)) * np.exp(-4.0 * np.arange(K) / K)   # a decaying row, as Lt
    B = rng.standard_normal((Nd, K))
    check(A, B, contraction(A, B), rng)


def test_wide_rows_zeros_and_coherent_sums():
    rng = np.random.default_rng(5)
    Md, Nd, K = 256, 512, 768
    A = rng.standard_normal((Md, K)) * 2.0 ** rng.integers(-40, 1, (Md, K))
    B = rng.standard_normal((Nd, K)) * 2.0 ** rng.integers(-300, 300, (Nd, 1))
    A[3] = 0.0
    A[5] = 1.9999999999999998       # every product alike: the levels reach their largest sums
    A[6] = -127.0 / 256 * (1 + 2.0 ** -8 + 2.0 ** -16 + 2.0 ** -24 + 2.0 ** -32 + 2.0 ** -40)
    B[5] = 1.9999999999999998
    B[6] = A[6, 0]
    B[7] = 5e-324
    A[8], B[8] = 1e-200, 1e-180     # the product underflows
    A[9, 1:] = 0.0
    C = contraction(A, B)
    check(A, B, C, rng)
    for i in (3, 5, 6, 8, 9):
        for j in (5, 6, 7, 8):
            exact = sum(Fraction(float(a)) * Fraction(float(b)) for a, b in zip(A[i], B[j]))
            bound = 2.0 ** -52 * abs(float(exact)) + K * 2.0 ** -57 * np.abs(A[i]).max() * np.abs(B[j]).max()
            assert abs(float(Fraction(float(C[j, i])) - exact)) <= bound + 5e-324


def test_not_finite_rows_stay_in_their_rows():
    rng = np.random.default_rng(6)
    Md, Nd, K = 200, 600, 300
    A, B = rng.standard_normal((Md, K)), rng.standard_normal((Nd, K))
    clean = contraction(A, B)
    A2, B2 = A.copy(), B.copy()
    B2[17, 5] = np.nan
    B2[40, 7] = np.inf
    A2[99, 8] = -np.inf
    C = contraction(A2, B2)
    keep_n, keep_m = np.ones(Nd, bool), np.ones(Md, bool)
    keep_n[[17, 40]] = keep_m[99] = False
    assert np.array_equal(C[np.ix_(keep_n, keep_m)], clean[np.ix_(keep_n, keep_m)])
    assert np.all(np.isnan(C[17]))
    assert np.array_equal(C[40, keep_m], np.inf * np.sign(A2[keep_m, 7]))
    assert np.array_equal(C[keep_n, 99], -np.inf * np.sign(B2[keep_n, 8]))
    assert np.array_equal(np.isnan(C[40, 99]), np.isnan(A2[99, 7] * np.inf - np.inf * B2[40, 8]))
