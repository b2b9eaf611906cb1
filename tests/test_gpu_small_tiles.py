"""Reduced-precision products of small tiles and ragged ends: parts of fewer than 64
rows (more or fewer than 32) and 32 columns (more or fewer than 16), inner lengths on
either side of the stages of 16, and several segments of a product in one chunk of
four stages (FP32-class) or not (emulated FP64); on both sides of the line between
products from planes and without.

Tolerances: the repository's bounds of the precisions, 1e-12 and 1e-5."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_19171_gb300 import workloads as W
from tests.gpu_helpers import need_gpu, rel_err, run_gpu

SHAPES = [(9, 1, 1, 0), (12, 1, 3, 2), (9, 2, 2, 1), (10, 5, 5, 3), (7, 15, 2, 17), (7, 16, 2, 16), (7, 17, 3, 15),
          (6, 31, 1, 33), (6, 31, 4, 20), (6, 32, 1, 32), (6, 32, 3, 16), (6, 33, 1, 1), (6, 33, 3, 20), (5, 47, 1, 16),
          (5, 48, 2, 16), (5, 49, 1, 15), (5, 63, 1, 63), (5, 64, 1, 16), (4, 64, 1, 64), (4, 65, 1, 17), (4, 80, 1, 31),
          (4, 128, 0, 128), (5, 64, 0, 40)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
def test_small_tiles(shape):
    need_gpu()
    M = W.random_arrowhead(*shape, seed=11 + shape[1])
    Lr, Sr, ldr = O.selinv(M)
    for precision, tol in ((1, 1e-12), (2, 1e-5)):
        for mode in ("fused", "split"):
            L, Sg, ld, status = run_gpu(M, mode, precision=precision)
            assert status[0] == 0
            assert rel_err(L, Lr) < tol and rel_err(Sg, Sr) < tol, (precision, mode)
            assert abs(ld - ldr) < tol * max(1.0, abs(ldr))
            for i in range(M.nt + (1 if M.a else 0)):
                assert np.array_equal(Sg[(i, i)], Sg[(i, i)].T)
