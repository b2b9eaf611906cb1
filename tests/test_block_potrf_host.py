"""The block POTRF on the host (no GPU): its own source, run by fibers in place
of threads (potrf_host.cpp). Its result may not depend on the order in which
the warps run between two block barriers, and is the Cholesky factor.

Tolerance: the factor of a block of order n with condition number near 1 is off
by a few n units in the last place; 1e-13 of the largest entry."""
import ctypes
import os
import shutil
import subprocess

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
