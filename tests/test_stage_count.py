"""The count of staging slots used by a CTA over a launch of any length: a stage's
slot, the parity of its barrier's phase and whether an earlier stage used the slot
are those of the exact count."""
import ctypes
import random

from tests.host_build import plan_host


def test_slots_and_phases_over_long_launches():
    lib, r = plan_host(), random.Random(0)
    lib.stages_run.restype, lib.stages_run.argtypes = ctypes.c_uint, [ctypes.c_uint] * 2
    for slots in (4, 8):
        kept, exact = 0, 0
        for step in range(40000):
            used = r.choice([1, 2, 7, 8, 64, 65, 4352, 1 << 20])
            for g in (0, used - 1):
                a, b = kept + g, exact + g
                assert a % slots == b % slots and a // slots % 2 == b // slots % 2 and (a >= slots) == (b >= slots)
                assert a < 1 << 32
            kept, exact = lib.stages_run(kept, used), exact + used
        assert exact > 1 << 32
