"""Block sizes and pivot ranges of the block kernels on the GPU.

The block POTRF works in panels of four columns with up to three warps per
panel, FP64 products in 16 x 16, 32 x 32 or 64 x 64 parts with their padding
left out, and the factor's triangular solves in parts of 8 or 16 rows: the
sizes here sit on either side of those edges. Tolerance: the FP64 parity bound
of the other tests (1e-10 of the largest entry)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_19171_gb300 import workloads as W
from tests.gpu_helpers import FP64_TOL, need_gpu, rel_err, run_gpu

# (nt, b, w, a): panel edges (multiples of 4, 28 and 56 rows below a panel),
# part edges (8, 16, 32, 64), ragged second blocks, arrows below and above them
SIZES = [(4, b, 1, a) for b, a in [(1, 1), (3, 4), (4, 5), (5, 0), (8, 9), (15, 16), (16, 17), (17, 3), (28, 31),
                                   (31, 32), (32, 33), (33, 7), (36, 15), (59, 60), (60, 61), (63, 64), (64, 65),
                                   (65, 48), (80, 8), (127, 20), (129, 1)]] + [(30, 48, 4, 40), (3, 300, 2, 70)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SIZES)
def test_block_size_edges(shape):
    M = W.random_arrowhead(*shape, seed=7 + shape[1])
    Lr, Sr, ldr = O.selinv(M)
    for mode in ("fused", "split"):
        L, S, ld, status = run_gpu(M, mode)
        assert status[0] == 0
        assert rel_err(L, Lr) < FP64_TOL and rel_err(S, Sr) < FP64_TOL
        assert abs(ld - ldr) < FP64_TOL * max(1.0, abs(ldr))


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [2.0 ** -1050, 2.0 ** -1022, 2.0 ** -500, 2.0 ** 900, 2.0 ** 1020])
def test_pivot_range(scale):
    """Pivots over the whole range of doubles, the subnormal ones (whose
    reciprocal overflows) and those above 2^1020 (whose reciprocal is
    subnormal) included: a block-diagonal matrix D with entries 1, 4, 16, 64
    times a power of four has the exact factor sqrt(D). Each entry passes one
    reciprocal square root and one product: 4 units in the last place."""
    need_gpu()
    nt, b = 2, 10
    M = W.random_arrowhead(nt, b, 0, 0, seed=0)
    scale = 2.0 ** (2 * int(np.log2(scale) // 2))
    d = np.array([1.0, 1.0, 0.25, 1.0, 0.0625, 0.25, 1.0, 0.25, 0.0625, 1.0]) * scale
    for k in range(nt):
        M.tiles[(k, k)] = np.diag(d)
    L, _, _, status = run_gpu(M, "split")
    assert status[0] == 0
    for k in range(nt):
        got = np.diag(L[(k, k)])
        assert np.all(np.abs(got / np.sqrt(d) - 1.0) <= 4 * 2.0 ** -53), got / np.sqrt(d) - 1.0
        assert np.all(np.tril(L[(k, k)], -1) == 0.0)
