"""Matrices whose pivots are powers of two while the entries below them in the
block are not zero: unit-diagonal (correlation) matrices, an AR(1) precision
with rho = 1/2 (every pivot is 1) and the (-1, 2, -1) stencil; and blocks
scaled so that some pivots lie outside the range of the block POTRF's integer
reciprocal. Every precision; solo (both forms), batched and served.

Tolerance: the repository's bound of each precision (FP64 1e-10, emulated FP64
1e-12, FP32-class 1e-5), or 8 x condition number x unit roundoff where that is
more."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_19171_gb300 import workloads as W
from tests.gpu_helpers import need_gpu, rel_err, run_gpu
from tests.test_block_potrf_host import scaled_block

BASE = {0: 1e-10, 1: 1e-12, 2: 1e-5}
ROUNDOFF = {0: 2.0 ** -53, 1: 2.0 ** -53, 2: 2.0 ** -24}
PRECISIONS = [0, 1, 2]


def matrix(kind, b, nt=4, a=5):
    n = nt * b + a
    if kind == "ar1":
        A = W.ar1_precision(n, 0.5)
    elif kind == "stencil":
        A = 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
    else:
        A = W.random_arrowhead(nt, b, 1, a, seed=b).to_dense()
        d = 1.0 / np.sqrt(np.diag(A))
        A = A * d[:, None] * d[None, :]
        np.fill_diagonal(A, 1.0)
    return W.ArrowheadTiles.from_dense(A, nt, b, 1, a), np.linalg.cond(A)


def bound(precision, cond):
    return max(BASE[precision], 8 * cond * ROUNDOFF[precision])


@pytest.mark.gpu
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("b", [4, 64, 100])
@pytest.mark.parametrize("kind", ["unit", "ar1", "stencil"])
def test_solo(kind, b, precision):
    need_gpu()
    M, cond = matrix(kind, b)
    tol = bound(precision, cond)
    Lr, Sr, ldr = O.selinv(M)
    for mode in ("fused", "split"):
        L, Sg, ld, status = run_gpu(M, mode, precision=precision)
        assert status[0] == 0
        assert rel_err(L, Lr) < tol and rel_err(Sg, Sr) < tol
        assert abs(ld - ldr) < tol * max(1.0, abs(ldr))


@pytest.mark.gpu
@pytest.mark.parametrize("precision", PRECISIONS)
def test_batch(precision):
    S = need_gpu()
    import torch
    mats = [matrix(kind, b) for kind, b in (("unit", 64), ("ar1", 100), ("stencil", 4))]
    bt = S.StilesBatch([(M.nt, M.b, M.w, M.a) for M, _ in mats], wait_budget_s=5.0, precision=precision)
    try:
        bt.upload([M for M, _ in mats]).factor_selinv()
        torch.cuda.synchronize()
        lds = bt.logdet()
        for m, (M, cond) in enumerate(mats):
            assert bt.status(m) == (0, 0)
            _, Sr, ldr = O.selinv(M)
            assert rel_err(bt.sigma_tiles(m), Sr) < bound(precision, cond)
            assert abs(lds[m] - ldr) < bound(precision, cond) * max(1.0, abs(ldr))
    finally:
        bt.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", PRECISIONS)
def test_served(precision):
    S = need_gpu()
    import time
    import torch
    M, cond = matrix("ar1", 100)
    shape = (M.nt, M.b, M.w, M.a)
    lay = S.PackedLayout(*shape)
    srv = S.StilesServer([shape], 1 << 24, max_requests=2, precision=precision)
    try:
        srv.set_base(0, torch.zeros(lay.doubles, dtype=torch.float64), *[torch.zeros(M.n, dtype=torch.float64)] * 2)
        srv.start(20.0)
        r = srv.submit_values(0, lay.pack(M.tiles, np.zeros(lay.doubles)))
        assert r is not None
        t0 = time.time()
        while not srv.poll():
            assert time.time() - t0 < 20.0
        code, _, ld = srv.result(r)
        out = torch.empty(lay.doubles, dtype=torch.float64)
        srv.sigma(r, out)
        srv.release(r)
        assert srv.stop() == S.STILES_OK and code == S.STILES_OK
        _, Sr, ldr = O.selinv(M)
        assert rel_err(lay.unpack(out.numpy()), Sr) < bound(precision, cond)
        assert abs(ld - ldr) < bound(precision, cond) * max(1.0, abs(ldr))
    finally:
        srv.close()


@pytest.mark.gpu
@pytest.mark.parametrize("b", [10, 41, 64])
@pytest.mark.parametrize("exponent", [-1040, -1022, 1019, 1021])
def test_scaled_blocks(b, exponent):
    """A = D B D, D a power of two per row: L = D chol(B), pivots around
    2^exponent, inside and outside the reciprocal's range, in one panel too."""
    need_gpu()
    A, unscale, ref, tol = scaled_block(b, exponent)
    M = W.ArrowheadTiles(2, b, 0, 0, {(0, 0): A, (1, 1): A})
    L, _, _, status = run_gpu(M, "split")
    assert status[0] == 0
    for k in range(2):
        assert np.abs(unscale(L[(k, k)]) - ref).max() <= tol
