"""The per-part trace: four whole records per task, whatever the number of its
parts, exactly one of them that of the part that completed the task."""
import ctypes

import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_19171_gb300 import workloads as W
from tests.gpu_helpers import FP64_TOL, need_gpu, rel_err
from tests.host_build import plan_host


def test_records_of_sixteen_parts():
    rec = np.arange(1, 65, dtype=np.uint64).reshape(16, 4)
    rec[:, 3] = 5
    rec[6, 2] = 500   # the last of parts 2, 6, 10, 14 to end
    rec[9, 3] |= 512  # completed the task
    out = np.zeros((4, 4), dtype=np.uint64)
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    plan_host().trace_pick(ptr(rec), ptr(out))
    assert np.array_equal(out, rec[[12, 9, 6, 15]])


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(16, 64, 1, 16), (12, 100, 2, 37)])
def test_every_task_has_whole_records(shape):
    S = need_gpu()
    import torch
    M = W.random_arrowhead(*shape, seed=2)
    st = S.Stiles(*shape, wait_budget_s=5.0).upload(M)
    try:
        S.stiles_set_option(st.h, S.STILES_OPT_TRACE, 1)
        for _ in range(3):
            st.factor_selinv()
            torch.cuda.synchronize()
            assert st.status()[0] == S.STILES_OK
            tr = S.stiles_trace(st.h)
            used = tr[..., 2] != 0
            assert np.all(used[:, 0]) and np.all(tr[..., 0][used] <= tr[..., 1][used])
            assert np.all(tr[..., 1][used] <= tr[..., 2][used])
            last = (tr[..., 3] >> np.uint64(9)) & np.uint64(1)
            assert np.all(last.sum(axis=1) == 1)
            op = tr[..., 3] & np.uint64(255)
            assert np.all((op == op[:, :1]) | ~used)
        _, Sr, _ = O.selinv(M)
        assert rel_err(st.sigma_tiles(), Sr) < FP64_TOL
    finally:
        st.close()
