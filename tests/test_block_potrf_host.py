"""The block POTRF on the host (no GPU): its own source, run by fibers in place
of threads (potrf_host.cpp). Its result may not depend on the order in which
the warps run between two block barriers, and is the Cholesky factor.

Tolerance: the factor of a block of order n with condition number near 1 is off
by a few n units in the last place; 1e-13 of the largest entry."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    so = str(tmp_path_factory.mktemp("potrf") / "potrf_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2504_19171_gb300", "csrc"), os.path.join(ROOT, "tests", "potrf_host.cpp"),
                    "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.recip_host.restype = ctypes.c_double
    lib.recip_host.argtypes = [ctypes.c_double, ctypes.c_int]
    return lib


def factor(lib, A, order=3210):
    n = A.shape[0]
    A = np.asfortranarray(A)
    L, rcp = np.zeros((n, n), order="F"), np.zeros(n)
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    assert lib.potrf_host(ptr(A), n, order, ptr(L), ptr(rcp)) == 0
    return L, rcp


def spd(n, seed):
    G = np.random.default_rng(seed).standard_normal((n, n))
    return G @ G.T / n + 2.0 * np.eye(n)


# panels of 4 columns; 28 rows below a panel's own per warp, up to three warps
@pytest.mark.parametrize("n", [1, 4, 5, 31, 32, 33, 36, 60, 61, 64])
def test_order_of_the_warps_does_not_matter(host, n):
    A = spd(n, n)
    ref = np.linalg.cholesky(A)
    L0, rcp0 = factor(host, A)
    assert np.abs(L0 - ref).max() <= 1e-13 * np.abs(ref).max()
    assert np.abs(rcp0 * np.diag(ref) - 1.0).max() <= 1e-13
    for order in (123, 1302, 2031, 321):  # digits from the last: warp 3 first, .., warp 0 last, and others
        L, rcp = factor(host, A, order)
        assert np.array_equal(L, L0) and np.array_equal(rcp, rcp0), order


def exact_error_ulp(r, d):
    """|r - 1/d| in units of the last place of the result, in exact arithmetic."""
    exact = 1 / abs(Fraction(d))
    return float(abs(Fraction(r) - exact) / Fraction(np.spacing(float(exact))))


@pytest.mark.parametrize("ulp", [-2, -1, 0, 1, 2])
def test_reciprocal(host, ulp):
    """Powers of two, their neighbours, values just below 2 and random ones, over
    the exponents of the range; the single-precision estimate off by `ulp` units."""
    rng = np.random.default_rng(0)
    ms = [1.0, np.nextafter(1.0, 2.0), 1.0 + 2.0 ** -29, 1.0 + 2.0 ** -23, 1.5, 2.0 - 2.0 ** -22, 2.0 - 2.0 ** -29,
          np.nextafter(2.0, 1.0)] + list(1.0 + rng.random(3000)) + list(1.0 + 2.0 ** rng.uniform(-52, 0, 500))
    for i, m in enumerate(ms):
        for e in (0, 1, -1, int(rng.integers(-1022, 1021)), -1022, 1020)[:6 if i < 8 else 4]:
            d = float(np.ldexp(m, e)) * (-1.0 if i % 3 == 1 else 1.0)
            r = host.recip_host(d, ulp)
            assert r > 0.0 and (exact_error_ulp(r, d) == 0.0 if m == 1.0 else exact_error_ulp(r, d) <= 0.51), (m, e, r)


def correlation(n):
    A = spd(n, n)
    d = 1.0 / np.sqrt(np.diag(A))
    A = A * d[:, None] * d[None, :]
    np.fill_diagonal(A, 1.0)
    return A


@pytest.mark.parametrize("n", [2, 4, 33, 64])
def test_pivots_that_are_powers_of_two(host, n):
    """A unit diagonal, an AR(1) precision with rho = 1/2 (every pivot 1) and the
    (-1, 2, -1) stencil (first pivot 2; condition number below 0.5 n^2)."""
    ar1 = 1.25 * np.eye(n) - 0.5 * (np.eye(n, k=1) + np.eye(n, k=-1))
    ar1[0, 0] = ar1[-1, -1] = 1.0
    stencil = 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
    for A in (correlation(n), ar1, stencil):
        ref = np.linalg.cholesky(A)
        L, rcp = factor(host, A)
        assert np.abs(L - ref).max() <= 1e-13 * np.abs(ref).max()
        assert np.abs(rcp * np.diag(ref) - 1.0).max() <= 1e-13 * n


@pytest.mark.parametrize("b", [10, 41, 64])
@pytest.mark.parametrize("exponent", [-1040, -1022, 1019, 1021])
def test_pivots_outside_the_range(host, b, exponent):
    A, unscale, ref, tol = scaled_block(b, exponent)
    for order in (3210, 123):
        L, _ = factor(host, A, order)
        assert np.abs(unscale(L) - ref).max() <= tol


def scaled_block(b, exponent):
    """(A, a factor's rows back to scale 1, chol(B), tolerance) for A = D B D
    with D_i = 2^e_i, 2 e_i within 4 of the exponent. An operation on entries of
    A loses at most 2^-1075 beside its roundoff, relative to the smallest scale
    2^(exponent - 4 - 1), and an entry takes part in b of them, grown by at most
    8: 64 b (2^-53 + 2^(-1070 - exponent))."""
    rng = np.random.default_rng(b)
    G = rng.standard_normal((b, b))
    e = np.minimum(exponent // 2 + rng.integers(-2, 2, b), 511)
    A = np.ldexp(np.eye(b) + 0.25 * (G @ G.T) / b, e[:, None] + e[None, :])
    ref = np.linalg.cholesky(np.ldexp(A, -e[:, None] - e[None, :]))  # of the matrix as stored
    return A, lambda L: np.ldexp(L, -e[:, None]), ref, 64 * b * (2.0 ** -53 + 2.0 ** (-1070 - exponent))
