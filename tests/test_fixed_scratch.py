"""Shapes at the edge of the allocation-free call's fixed scratch array: those
whose finest-cut plan exceeds it by its queue slots alone run on a plan of fewer
parts, with the same results bit for bit."""
import ctypes

import pytest

from tests.gpu_helpers import need_gpu
from tests.host_build import plan_host

LIMIT = 64 << 20
SHAPES = [(509, 64, 2, 64), (407, 64, 4, 0), (339, 64, 4, 64), (301, 96, 2, 0), (365, 100, 0, 128), (194, 100, 2, 128),
          (127, 128, 2, 128), (104, 200, 1, 0)]


@pytest.mark.parametrize("shape", SHAPES)
def test_a_plan_fits(shape):
    most = ctypes.c_longlong()
    got = plan_host().fixed_scratch(*shape, 0, LIMIT, ctypes.byref(most))
    assert most.value > LIMIT and 0 < got <= LIMIT


def test_tiles_beyond_the_array_are_refused():
    most = ctypes.c_longlong()
    assert plan_host().fixed_scratch(520, 64, 2, 64, 0, LIMIT, ctypes.byref(most)) == -1


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(339, 64, 4, 64), (194, 100, 2, 128), (104, 200, 1, 0)])
def test_same_results(shape):
    S = need_gpu()
    import torch
    from paper_2504_19171_gb300 import workloads as W
    st = S.Stiles(*shape, wait_budget_s=10.0)
    try:
        assert S.stiles_workspace_bytes(st.h)[2] > LIMIT
        st.A = torch.zeros(st.doubles, dtype=torch.float64, device="cuda")
        W.random_arrowhead_packed(*shape, 3, st.A)
        st.L.zero_()
        st.S.zero_()
        st.factor_selinv()
        torch.cuda.synchronize()
        assert st.status()[0] == S.STILES_OK
        ld = st.logdet()
        L, Sg = torch.zeros_like(st.L), torch.zeros_like(st.S)
        S.stiles_factor_selinv_noalloc(st.h, st.A.data_ptr(), L.data_ptr(), Sg.data_ptr(), st.stream_ptr())
        torch.cuda.synchronize()
        assert st.status()[0] == S.STILES_OK and S.stiles_logdet(st.h) == (S.STILES_OK, ld)
        assert torch.equal(L, st.L) and torch.equal(Sg, st.S)
    finally:
        st.close()
