"""The backward recurrence of the Bessel functions (csrc/hankel.cuh) with its start from a
table, compiled for the host.  The table holds 0 where the kernel that wrote it evaluated an
argument outside the recurrence's range; an evaluation that differs in the last bit may
still enter it, at the ends of the range 2 .. 17."""

import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest
from scipy.special import jv, yv

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if gxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers not found")
    so = str(tmp_path_factory.mktemp("rec") / "recurrence.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + inc, "-o", so,
                    os.path.join(HERE, "recurrence_start_check.cpp")], check=True, capture_output=True, timeout=300)
    return C.CDLL(so)


@pytest.mark.parametrize("x", [np.nextafter(2.0, 3.0), 2.5, 11.99, 12.0, 17.0])
@pytest.mark.parametrize("tabulated", [0, None, 70])
def test_recurrence_from_a_table(lib, x, tabulated):
    start = lib.recurrence_start(C.c_double(x)) if tabulated is None else tabulated
    out = np.zeros(4)
    lib.recurrence_from(C.c_double(x), start, out.ctypes.data_as(C.c_void_p))
    want = np.array([jv(0, x), jv(1, x), yv(0, x), yv(1, x)])
    assert np.max(np.abs(out - want)) < 2e-13        # the branch's own accuracy
