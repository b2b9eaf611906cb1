"""Memory of the planes (the reduced precisions' split operands): a ring of
band + 1 tile columns of Sigma, each with the diagonal tile, `band` band tiles and
the arrow by columns, and all but one of them by rows, two columns of U, and the
corner; none for a matrix that fills the device."""
import pytest

from paper_2504_19171_gb300 import stiles as S
from tests.host_build import plan_host


def group(prec, k):
    return -(-k // 16) * 2048 * (8 if prec == 1 else 3) + (256 * -(-k // 512) if prec == 1 else 0)


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("shape", [(6, 1024, 4, 64), (20, 1024, 10, 64), (200, 1024, 1, 64), (40, 100, 2, 37), (9, 33, 4, 20),
                                   (5, 160, 3, 0)])
def test_ring(shape, prec):
    nt, b, w, a = shape
    R, ra = -(-b // 64), -(-a // 64)
    tile, arrow, arrow_rows = R * group(prec, b), R * group(prec, a) if a else 0, ra * group(prec, b)
    column = 2 * w * tile + arrow + arrow_rows  # diagonal, w by columns, w - 1 by rows
    want = (w + 1) * column + 2 * (w * tile + arrow) + (ra * group(prec, a) if a else 0)
    assert plan_host().plane_bytes(*shape, prec) == want
    for kind in (S.PLAN_SELINV, S.PLAN_FUSED):
        small = (min(nt, w + 4), min(b, 192), w, a) if w < 5 else (8, 80, 6, 9)
        assert S.stiles_debug_validate(*small, kind, prec) == S.STILES_OK
        assert S.stiles_debug_race_check(*small, kind, prec) == S.STILES_OK


def test_short_wide_matrix():
    """(6, 1024, 4, 64) in emulated FP64: 1.05 GB with a ring of band + 2 columns of
    2 band + 1 tiles."""
    assert plan_host().plane_bytes(6, 1024, 4, 64, 1) < 0.86e9


def test_a_matrix_that_fills_the_device_has_none():
    fit = plan_host().planes_go_in
    device = 284 << 30
    packed = device // 4 // 8  # four buffers of it are the device
    assert not fit(packed, 1 << 30, device)
    assert not fit(int(0.93 * packed), 5 << 30, device) and fit(int(0.93 * packed), 1 << 30, device)


@pytest.mark.parametrize("prec", [1, 2])
def test_which_shapes_take_planes(prec):
    """With a band, from an inner length (w b + a) of 112 and a tile order of 24
    (FP32-class) or 32 (emulated FP64) on; in emulated FP64 with tiles below 64 for arrows
    of up to 64 only (no tile's K beyond one exponent of either kind of part)."""
    takes = lambda *shape: plan_host().plane_faults(*shape, prec, 0) == 0
    assert all(takes(*s) for s in [(6, 32, 3, 16), (6, 64, 1, 48), (6, 48, 2, 16), (6, 112, 1, 0), (6, 63, 1, 64), (6, 64, 1, 65)])
    assert not any(takes(*s) for s in [(6, 23, 3, 64), (6, 32, 3, 15), (6, 64, 1, 47), (6, 128, 0, 512)])
    assert all(takes(*s) == (prec == 2) for s in [(6, 24, 3, 40), (6, 31, 3, 40), (6, 63, 1, 65)])
