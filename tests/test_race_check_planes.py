"""Race check of the planes' exponents: a group of emulated FP64 begins with the
exponents of its vectors (16 units of 16 bytes per 512 of K), which its split writes
and its products read."""
import pytest

from paper_2504_19171_gb300 import stiles as S
from tests.host_build import plan_host


@pytest.mark.parametrize("prec,head,stages", [(1, 16, 1024), (2, 0, 384)])
def test_unordered_splits(prec, head, stages):
    check = plan_host().two_splits
    assert check(prec, head + stages) == S.STILES_OK             # side by side
    assert check(prec, head + stages - 16) == S.STILES_ERR_PLAN  # one's last stages over the other's first units (its exponents)
