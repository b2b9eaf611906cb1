"""Statistics of a batch's merged plan: every field, the list schedule's makespan
among them, is that of the plan."""
import pytest

from tests.gpu_helpers import need_gpu


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [0, 1])
def test_batch_statistics(precision):
    S = need_gpu()
    shapes = [(6, 64, 1, 16), (5, 100, 2, 37), (8, 128, 1, 20)]
    bt = S.StilesBatch(shapes, precision=precision)
    try:
        st = S.stiles_batch_stats(bt.h)
        solo = [S.stiles_plan_stats(*sh, S.PLAN_FUSED, 304, precision) for sh in shapes]
        # flops are stated per matrix in whole numbers
        assert abs(st["flops"] - sum(x["flops"] for x in solo)) <= len(shapes)
        assert st["critical_path_ns"] >= max(x["critical_path_ns"] for x in solo) - 1
        assert st["makespan_ns"] >= st["critical_path_ns"] > 0
        assert S.stiles_batch_stats(bt.h) == st
    finally:
        bt.close()
