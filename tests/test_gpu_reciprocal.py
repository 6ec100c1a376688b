"""reciprocal(), on which forces and the objective stand, against the IEEE
reciprocal: every float from 1 to infinity, and NaN."""
import ctypes
import os
import subprocess

import pytest

from paper_2608_01907_gb300 import _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_reciprocal_equals_ieee_over_its_whole_range(cuda, tmp_path):
    lib = str(tmp_path / "reciprocal_check.so")
    subprocess.run([_build._nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                    _build.CSRC, os.path.join(HERE, "reciprocal_check.cu"), "-o", lib], check=True)
    out = (ctypes.c_ulonglong * 3)(1, 1, 1)
    assert ctypes.CDLL(lib).compare_reciprocals(out) == 0
    assert list(out) == [0, 0, 0]
