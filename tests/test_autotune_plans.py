"""The autotuner times a plan once: codes that differ only in the phase-2 split give
the same plan in the reduced precisions."""
import pytest

from paper_2504_19171_gb300 import autotune as AT
from paper_2504_19171_gb300 import stiles as S


class Fake:
    """A batch handle that counts the codes it is built with."""
    built = []

    def __init__(self, shapes, device=None, precision=0, tuning=None):
        Fake.built.append(tuning[0])
        raise RuntimeError("no GPU")


@pytest.mark.parametrize("precision,want", [(S.STILES_FP64, 8), (S.STILES_EMU64, 5), (S.STILES_FP32X, 5)])
def test_distinct_plans(precision, want):
    codes = {AT.same_plan_as(c, precision) for c in AT.CANDIDATES}
    assert len(codes) == want and 0 in codes
    for c in AT.CANDIDATES:  # the stand-in has the plan of the code (statistics of every kind)
        for shape in ((12, 256, 2, 60), (6, 48, 1, 9), (12, 1024, 1, 64)):
            a, b = (S.stiles_plan_stats(*shape, S.PLAN_FUSED + 256 * x, 304, precision)
                    for x in (c, AT.same_plan_as(c, precision)))
            assert a == b


def test_a_plan_is_timed_once(monkeypatch):
    monkeypatch.setattr(AT.S, "StilesBatch", Fake)
    t = AT.Autotuner(candidates=(4, 8, 0))
    Fake.built.clear()
    with pytest.raises(RuntimeError):
        t.tune(64, 1, 8, S.STILES_EMU64)
    assert Fake.built == [0]
