"""Host (g++) builds of the library's sources for CPU tests."""
import ctypes
import functools
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2504_19171_gb300", "csrc")


@functools.lru_cache(maxsize=None)
def plan_host():
    """tests/plan_host.cpp with the planner, as a shared library."""
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    so = os.path.join(tempfile.mkdtemp(prefix="plan_host"), "plan_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, os.path.join(ROOT, "tests", "plan_host.cpp"),
                    os.path.join(CSRC, "plan.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.fixed_scratch.restype = ctypes.c_longlong
    lib.fixed_scratch.argtypes = [ctypes.c_int] * 5 + [ctypes.c_longlong, ctypes.POINTER(ctypes.c_longlong)]
    lib.plane_bytes.restype = ctypes.c_longlong
    lib.planes_go_in.argtypes = [ctypes.c_longlong] * 3
    return lib
