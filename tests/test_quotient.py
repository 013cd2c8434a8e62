"""The refinement's quotient (csrc/quotient.cuh), compiled for the host: equal to the
division over the stated range, near it below, and no number for an infinite
numerator."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include <cmath>
#define __device__
#define __forceinline__ inline
static float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
#include "quotient.cuh"
extern "C" void run(long n, const float *num, const float *det, float *q) {
    for (long i = 0; i < n; ++i) q[i] = quotient(num[i], det[i], 1.f / det[i]);
}
"""


@pytest.fixture(scope="module")
def quotient(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotient")
    (d / "q.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1501_02565_gb300", "csrc"), "-o", str(d / "q.so"), str(d / "q.cpp")],
                   check=True)
    run = ctypes.CDLL(str(d / "q.so")).run

    def call(num, det):
        num, det = np.ascontiguousarray(num, np.float32), np.ascontiguousarray(det, np.float32)
        out = np.empty(len(num), np.float32)
        run(ctypes.c_long(len(num)), *(ctypes.c_void_p(a.ctypes.data) for a in (num, det, out)))
        return out

    return call


def _divide(n, det):
    with np.errstate(all="ignore"):
        return np.asarray(n, np.float32) / np.asarray(det, np.float32)


def _random(rng, n, lo, hi):
    m = rng.integers(1 << 23, 1 << 24, n).astype(np.float64)
    m[: n // 8] = (1 << 24) - rng.integers(1, 3, n // 8)    # mantissas of ones
    m[n // 8: n // 4] = (1 << 23) + rng.integers(0, 3, n // 8)
    return (rng.permutation(m) * 2.0 ** (rng.integers(lo, hi, n) - 23)).astype(np.float32)


def test_equal_to_the_division_in_the_stated_range(quotient):
    rng = np.random.default_rng(1)
    n = 3000000
    det = _random(rng, n, -59, 59)   # (the refinement's: between 1e-18 and 1e18)
    num = _random(rng, n, -98, 99) * rng.choice([-1, 1], n)
    num[rng.random(n) < 0.05] = 0.0
    q = np.abs(_divide(num, det))
    num[(q != 0) & ((q < 2.0 ** -98) | (q > 2.0 ** 99))] = 1.0
    assert np.array_equal(quotient(num, det), _divide(num, det))


def test_near_the_division_below_it(quotient):
    rng = np.random.default_rng(2)
    n = 500000
    det, num = _random(rng, n, -59, 59), _random(rng, n, -126, -99)
    want = _divide(num, det)
    assert (np.abs(quotient(num, det).astype(np.float64) - want) <= np.spacing(want) + 2.0 ** -149).all()


def test_what_leaves_no_residual(quotient):
    assert np.isnan(quotient([np.inf, -np.inf, np.nan], [2.0, 3.0, 2.0])).all()
