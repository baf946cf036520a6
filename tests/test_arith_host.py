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
void quotients(const double* n, const double* d, long count, double* by, double* q)
{
    for (long i = 0; i < count; ++i) {
        by[i] = pdhg::div_by(n[i], d[i], 1.0 / d[i]);
        q[i] = pdhg::quotient(n[i], d[i]);
    }
}
// clamp, positive part, v > 0, lo < v < hi and the keys' order of v and lo
void compare(const double* v, const double* lo, const double* hi, long count, double* clamp,
             double* pos, int* positive, int* inside, int* below)
{
    for (long i = 0; i < count; ++i) {
        clamp[i] = pdhg::res_clamp(v[i], lo[i], hi[i]);
        pos[i] = pdhg::res_pos(v[i]);
        positive[i] = pdhg::res_positive(v[i]);
        inside[i] = pdhg::res_inside(v[i], lo[i], hi[i]);
        below[i] = pdhg::order_key(v[i]) < pdhg::order_key(lo[i]);
    }
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
    lib.quotients.argtypes = [C.c_void_p, C.c_void_p, C.c_long, C.c_void_p, C.c_void_p]
    lib.compare.argtypes = [C.c_void_p] * 3 + [C.c_long] + [C.c_void_p] * 5
    return lib


def _quotients(lib, n, d):
    n, d = np.ascontiguousarray(n, np.float64), np.ascontiguousarray(d, np.float64)
    by, q = np.empty_like(n), np.empty_like(n)
    lib.quotients(n.ctypes.data, d.ctypes.data, n.size, by.ctypes.data, q.ctypes.data)
    return by, q


def test_largest_of_values_that_are_not_negative(lib):
    """A -0 (a >= row that did not move) or a NaN beside a violated row hides nothing."""
    rng = np.random.default_rng(0)
    for _ in range(2000):
        v = rng.choice(SPECIAL[:-1] + [np.nan, -0.0, 1e-3], 32)
        got, want = lib.max_of(v.ctypes.data, 32), np.fmax.reduce(np.append(v, 0.0))
        assert got == want and not np.signbit(got)
    assert lib.max_of(np.array([3.0, np.inf, -0.0, np.nan]).ctypes.data, 4) == np.inf


def _next_to_midpoints(rng, count):
    """Pairs of 53-bit integers whose quotient lies as close to the middle of two doubles as
    one can: n 2^s = d M +- 1 with an odd M of 54 bits, from the inverse of d modulo 2^s."""
    n, d = [], []
    while len(n) < count:
        dd = int(rng.integers(2 ** 52, 2 ** 53)) | 1
        for s in (53, 54):
            inv = pow(dd, -1, 2 ** s)
            for sign, M in ((-1, inv), (1, 2 ** s - inv)):
                nn = (dd * M + sign) >> s
                if 2 ** 53 <= M < 2 ** 54 and 2 ** 52 <= nn < 2 ** 53:
                    n.append(float(nn))
                    d.append(float(dd))
    return np.array(n), np.array(d)


def test_quotients_are_the_divisions(lib):
    rng = np.random.default_rng(1)
    n, d = 1.0 + rng.random(200000), 1.0 + rng.random(200000)
    pairs = [(n, d), (n * 2.0 ** rng.integers(-100, 101, n.size), d * 2.0 ** rng.integers(-90, 91, n.size)),
             _next_to_midpoints(rng, 40000)]
    # mantissas of almost all ones and almost all zeros
    ends = np.concatenate([2.0 ** 53 - np.arange(1, 60), 2.0 ** 52 + np.arange(60)])
    pairs.append(tuple(v.ravel() for v in np.meshgrid(ends, ends)))
    for n, d in pairs:
        by, q = _quotients(lib, n, d)
        assert np.array_equal(by, n / d) and np.array_equal(q, n / d)


def test_quotient_beyond_its_range_divides(lib):
    edge = [2.0 ** -101, 2.0 ** -100, 2.0 ** 100, 2.0 ** 101, 5e-324, 1e-300, 1e300, 0.0, np.inf]
    nums = np.array([0.0, 1.0, 3.0, 2.0 ** -501, 2.0 ** -500, 2.0 ** 500, 2.0 ** 501, 5e-324, 1e308, np.inf,
                     np.nan])
    with np.errstate(all="ignore"):
        for d in edge:
            dd = np.full(nums.size, d)
            assert np.array_equal(_quotients(lib, nums, dd)[1], nums / dd, equal_nan=True)


def test_comparisons_on_bit_patterns(lib):
    vals = np.array(SPECIAL + [-v for v in SPECIAL] + [np.nan, 0.5, -0.5, -1.0 - 2.0 ** -52])
    bounds = np.array([v for v in vals if not np.isnan(v)])
    v, lo, hi = (a.ravel() for a in np.meshgrid(vals, bounds, bounds))
    keep = lo <= hi
    v, lo, hi = (np.ascontiguousarray(a[keep]) for a in (v, lo, hi))
    clamp, pos = np.empty_like(v), np.empty_like(v)
    flags = [np.empty(v.size, np.int32) for _ in range(3)]
    lib.compare(v.ctypes.data, lo.ctypes.data, hi.ctypes.data, v.size, clamp.ctypes.data,
                pos.ctypes.data, *(f.ctypes.data for f in flags))
    positive, inside, below = flags
    want = np.where(v < lo, lo, v)
    want = np.where(want > hi, hi, want)
    assert np.array_equal(clamp, want, equal_nan=True)     # (the zeros are equal)
    assert np.array_equal(pos, np.where(v < 0.0, 0.0, v), equal_nan=True)
    assert np.array_equal(positive != 0, v > 0.0)
    assert np.array_equal(inside != 0, (lo < v) & (v < hi))
    some = ~np.isnan(v) & (v != lo)
    assert np.array_equal(below[some] != 0, v[some] < lo[some])
