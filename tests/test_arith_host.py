"""Arithmetic on bit patterns (csrc/arith.cuh), compiled for the host: the same source
that the kernels compile, against plain comparisons and divisions."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2508_16806_gb300", "csrc")
HARNESS = r"""
#include "arith.cuh"
extern "C" {
double max_of(const double* v, long n)
{
    unsigned long long b = 0;
    for (long i = 0; i < n; ++i) {
        const unsigned long long k = pdhg::nonneg_key(v[i]);
        b = k > b ? k : b;
    }
    return pdhg::bits_double((long long)b);
}
}
"""
SPECIAL = [0.0, -0.0, 5e-324, 2.2e-308, 2.3e-308, 1.0, 1.0 + 2.0 ** -52, 1e300, 1.7976931348623157e308,
           np.inf]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    src, out = d / "arith.cpp", d / "arith.so"
    src.write_text(HARNESS)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                           "-I", CSRC, "-o", str(out), str(src), "-lm"])
    lib = C.CDLL(str(out))
    lib.max_of.argtypes, lib.max_of.restype = [C.c_void_p, C.c_long], C.c_double
    return lib


def test_largest_of_values_that_are_not_negative(lib):
    """A -0 (a >= row that did not move) or a NaN beside a violated row hides nothing."""
    rng = np.random.default_rng(0)
    for _ in range(2000):
        v = rng.choice(SPECIAL[:-1] + [np.nan, -0.0, 1e-3], 32)
        got, want = lib.max_of(v.ctypes.data, 32), np.fmax.reduce(np.append(v, 0.0))
        assert got == want and not np.signbit(got)
    assert lib.max_of(np.array([3.0, np.inf, -0.0, np.nan]).ctypes.data, 4) == np.inf
