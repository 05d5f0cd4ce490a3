"""The fixed-point Box-Muller normal of the critical-value simulation
(csrc/lambda_fixed.cuh) on the host, against 50-digit decimal arithmetic.

The function returns |z| / sqrt(2).  Bound: -ln u is truncated to 2^-58 in three
terms, so its root is off by at most 2^-56.4 / 2 / 2^-6 where u < 1 - 2^-12;
nearer to 1 the logarithm is FP64, 2^-53 relative.  The cosine and the product
add a few 2^-59: 2^-51 in all, the rounding of an FP64 value of magnitude 4.
"""
import ctypes
import os
import random
import subprocess
from decimal import Decimal, getcontext

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#define __host__
#define __device__
#define __forceinline__ inline
#include "lambda_fixed.cuh"
extern "C" long long normal_q59(unsigned long long n, unsigned long long f) {
    using namespace bfm::fixedpt;
    static uint64_t ln[256];
    static uint32_t rec[256];
    if (!rec[0])
        for (uint32_t i = 0; i < 256; ++i) {
            ln[i] = log_entry(i);
            rec[i] = log_recip(i);
        }
    bool neg;
    const uint64_t z = normal_q59(n, f, ln, rec, neg);
    return neg ? -(long long)z : (long long)z;
}
"""
PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494")


@pytest.fixture(scope="module")
def normal(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "n.cpp").write_text(SRC)
    so = str(d / "n.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_1807_01751_gb300", "csrc"), str(d / "n.cpp"), "-o", so])
    f = ctypes.CDLL(so).normal_q59
    f.argtypes, f.restype = [ctypes.c_uint64, ctypes.c_uint64], ctypes.c_int64
    return f


def cosine(x):
    term, total, k = Decimal(1), Decimal(1), 0
    while abs(term) > Decimal(10) ** -40:
        k += 2
        term *= -x * x / (k * (k - 1))
        total += term
    return total


def test_normals(normal):
    getcontext().prec = 50
    r = random.Random(5)
    top = 2 ** 53
    ns = [1, 2, 3, top, top - 1, top - 2, top // 2, top // 2 + 1, top // 2 - 1, top - 2 ** 41, top - 2 ** 41 + 1,
          top - 2 ** 41 - 1]
    ns += [max(1, r.randrange(top) >> r.randrange(53)) for _ in range(200)]
    ns += [top - (r.randrange(top) >> r.randrange(53)) for _ in range(200)]
    ns += [r.randrange(1, top + 1) for _ in range(400)]
    fs = [0, 1, top - 1] + [q * top // 8 + e for q in range(1, 8) for e in (-1, 0, 1)]
    total = Decimal(0)
    for i, n in enumerate(ns):
        f = fs[i % len(fs)] if i % 3 == 0 else r.randrange(top)
        x = Decimal(f) / top
        ref = (-(Decimal(n) / top).ln()).sqrt() * cosine(2 * PI * (x if x <= Decimal(0.5) else 1 - x))
        err = abs(Decimal(normal(n, f)) / 2 ** 59 - ref)
        assert err <= Decimal(2) ** -51, (n, f, float(err))
        total += err
    assert total / len(ns) < Decimal(2) ** -55
