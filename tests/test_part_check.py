"""The check that the self-checking device build makes of every task part before it
runs (and the host of whole tables), on the tasks that work on planes: their planes,
sources, outputs, input and mirror blocks."""
import pytest

from tests.host_build import plan_host


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("shape", [(5, 128, 2, 24), (4, 192, 1, 40)])
def test_planted_faults_are_found(shape, prec):
    find = plan_host().plane_faults
    assert find(*shape, prec, 0) == 0
    for which in range(1, 8):
        assert find(*shape, prec, which) > 0, which
