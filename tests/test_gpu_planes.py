"""Reduced-precision products from pre-split planes (phase 2, inner length 112
and up) and in self-splitting 64 x 32 parts, at the edges of their layout: vector
groups of 64, column halves of 32, stages of 16 and chunks of 512 of K (256 per
drain), the ring of plane slots (more tile columns than bandwidth + 2), tiles by
rows as well as by columns (bandwidth 2 and more), arrows of one and two groups.

Tolerances, derived before the first run: emulated FP64 the repository's 1e-12;
FP32-class products are off by a few 2^-24 of their largest terms and at most
eight tile columns are chained here: 1e-5."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_19171_gb300 import stiles as S
from paper_2504_19171_gb300 import workloads as W
from tests.gpu_helpers import need_gpu, rel_err, run_gpu

SHAPES = [(8, 127, 1, 9), (8, 128, 1, 16), (7, 129, 1, 0), (6, 144, 2, 33), (7, 160, 3, 1), (5, 192, 2, 70),
          (3, 272, 1, 65), (3, 528, 1, 17), (4, 130, 0, 20), (9, 64, 2, 31)]


@pytest.mark.parametrize("precision", [S.STILES_EMU64, S.STILES_FP32X])
@pytest.mark.parametrize("shape", [(6, 128, 1, 16), (5, 129, 2, 0), (4, 144, 3, 33), (3, 192, 0, 70), (4, 160, 2, 1)])
def test_plane_tables(shape, precision):
    """Host: every access in bounds and ordered (planes and their ring slots included)."""
    for kind in (S.PLAN_SELINV, S.PLAN_FUSED):
        assert S.stiles_debug_validate(*shape, kind, precision) == S.STILES_OK
        assert S.stiles_debug_race_check(*shape, kind, precision) == S.STILES_OK
    assert S.stiles_debug_race_check_serve(*shape, precision) == S.STILES_OK


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
def test_reduced_precisions(shape):
    need_gpu()
    M = W.random_arrowhead(*shape, seed=3 + shape[1])
    Lr, Sr, ldr = O.selinv(M)
    for precision, tol in ((S.STILES_EMU64, 1e-12), (S.STILES_FP32X, 1e-5)):
        for mode in ("fused", "split"):
            L, Sg, ld, status = run_gpu(M, mode, precision=precision)
            assert status[0] == 0
            assert rel_err(L, Lr) < tol and rel_err(Sg, Sr) < tol, (precision, mode)
            assert abs(ld - ldr) < tol * max(1.0, abs(ldr))
            for i in range(M.nt + (1 if M.a else 0)):
                assert np.array_equal(Sg[(i, i)], Sg[(i, i)].T)


@pytest.mark.parametrize("shape", [(9, 64, 1, 47), (9, 64, 1, 48), (9, 63, 2, 64), (8, 65, 2, 1), (7, 100, 4, 9), (6, 112, 1, 0)])
def test_small_tile_tables(shape):
    """Host, both sides of the line between products with and without planes."""
    for kind in (S.PLAN_SELINV, S.PLAN_FUSED):
        assert S.stiles_debug_validate(*shape, kind, S.STILES_EMU64) == S.STILES_OK
        assert S.stiles_debug_race_check(*shape, kind, S.STILES_EMU64) == S.STILES_OK


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [S.STILES_EMU64, S.STILES_FP32X])
@pytest.mark.parametrize("nt", [20, 28])
def test_noalloc_without_planes(nt, precision):
    """Shapes whose tiles fit the fixed scratch but whose planes do not (but for
    the FP32-class planes of the shorter one): the allocation-free call takes
    products without planes. Both forms are within
    the precision's bound of the exact result, so within twice of each other."""
    need_gpu()
    import torch
    shape = (nt, 256, 3, 64)
    st = S.Stiles(*shape, precision=precision)
    try:
        fits = nt == 20 and precision == S.STILES_FP32X
        assert 8 * st.doubles <= S.NOALLOC_SCRATCH_BYTES
        assert (S.stiles_workspace_bytes(st.h)[2] <= S.NOALLOC_SCRATCH_BYTES) == fits
        st.A = torch.zeros(st.doubles, dtype=torch.float64, device="cuda")
        W.random_arrowhead_packed(*shape, 5, st.A)
        st.L.zero_()
        st.S.zero_()
        st.factor_selinv()
        ref, ld = st.S.clone(), st.logdet()
        L, Sg = torch.zeros_like(st.L), torch.zeros_like(st.S)
        for _ in range(2):
            S.stiles_factor_selinv_noalloc(st.h, st.A.data_ptr(), L.data_ptr(), Sg.data_ptr(), st.stream_ptr())
        torch.cuda.synchronize()
        assert st.status()[0] == S.STILES_OK
        rc, ld2 = S.stiles_logdet(st.h)
        tol = 2e-12 if precision == S.STILES_EMU64 else 2e-5
        assert rc == S.STILES_OK and abs(ld2 - ld) <= tol * abs(ld)
        assert (Sg - ref).abs().max() <= tol * ref.abs().max()
        assert (L - st.L).abs().max() <= tol * st.L.abs().max()
    finally:
        st.close()
