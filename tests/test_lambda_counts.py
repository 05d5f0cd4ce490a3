"""Loop counters of the critical-value simulation (csrc/lambda_fixed.cuh: Count) at the
largest numbers of steps and paths that an int holds: a strided loop from a stride
before the end ends, and visits no index at or beyond it."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#define __host__
#define __device__
#define __forceinline__ inline
#include "lambda_fixed.cuh"
using bfm::fixedpt::Count;
// the largest index that the loop visits from `first` on, -1 where it runs on
extern "C" long long last(int first, int n, int stride) {
    long long top = -2;
    int visits = 0;
    for (Count i = (Count)first; i < (Count)n; i += stride) {
        if (++visits > 3 || (long long)i < 0) return -1;
        top = (long long)i > top ? (long long)i : top;
    }
    return top;
}
"""


@pytest.fixture(scope="module")
def last(tmp_path_factory):
    d = tmp_path_factory.mktemp("counts")
    (d / "c.cpp").write_text(SRC)
    so = str(d / "c.so")
    subprocess.check_call(["g++", "-O1", "-fwrapv", "-std=c++17", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_1807_01751_gb300", "csrc"), str(d / "c.cpp"), "-o", so])
    f = ctypes.CDLL(so).last
    f.restype = ctypes.c_longlong
    return f


@pytest.mark.parametrize("stride", [64, 1024])  # steps of a warp, threads of the selection
@pytest.mark.parametrize("n", [2 ** 31 - 1, 2 ** 31 - 64, 2 ** 31 - 1025, 1000])
def test_strides_end(last, n, stride):
    for first in (n - 1, n - stride, n - stride - 1, n - 2 * stride + 1):
        if first >= 0:
            assert 0 <= last(first, n, stride) < n
