"""The training kernel's reciprocal against CUDA's division, for every float of its
range (tests/reciprocal_check.cu).  Bound: before its last rounding the result is
off by at most 2^-45 of itself, and floats lie 2^-24 of themselves apart or more,
so it rounds the other way for at most 2 * 2^-45 / 2^-24 = 2^-20 of the values if
their exact reciprocals are spread evenly, by one unit; ten times that is allowed."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_value_of_the_range(tmp_path):
    so = tmp_path / "libreciprocal.so"
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "paper_2502_09541_gb300", "csrc"),
                           "-o", str(so), os.path.join(ROOT, "tests", "reciprocal_check.cu")])
    values, differ, most, nan = ctypes.c_uint64(), ctypes.c_uint64(), ctypes.c_uint32(), ctypes.c_uint32()
    assert ctypes.CDLL(str(so)).reciprocal_check(ctypes.byref(values), ctypes.byref(differ), ctypes.byref(most),
                                                 ctypes.byref(nan)) == 0
    assert values.value > 900_000_000 and nan.value == 1
    assert most.value <= 1 and differ.value <= 10 * values.value / 2**20
