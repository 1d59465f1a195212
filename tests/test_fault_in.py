"""Faulting in the pages of a caller's array leaves its contents alone (CPU only).

The averages' arrays get one write per page before the device copies into
them; should the copy then fail, the caller still has the old contents.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from test_index_mutants import CSRC, cuda_include

SOURCE = '#include "%s"\nextern "C" void touch(void *p, size_t n) { lbm::fault_in(p, n); }\n'


@pytest.fixture(scope="module")
def touch(tmp_path_factory):
    d = tmp_path_factory.mktemp("fault_in")
    src, lib = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as fh:
        fh.write(SOURCE % os.path.join(CSRC, "lbm_internal.h"))
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", "-I" + cuda_include(), src, "-o", lib, "-ldl"],
                   check=True, capture_output=True)
    f = C.CDLL(lib).touch
    f.argtypes, f.restype = [C.c_void_p, C.c_size_t], None
    return f


@pytest.mark.parametrize("n", [0, 1, 8, 4095, 4096, 4097, 100003])
def test_contents_survive(touch, n):
    a = np.random.default_rng(n).integers(1, 256, n + 64, dtype=np.uint8)
    b = a.copy()
    touch(b.ctypes.data + 5, n)
    assert np.array_equal(a, b)
