"""Conversions of the fixed-point transforms on the CPU: results are the nearest double
over the normal range, and below it, where FP64 arithmetic underflows gradually, within
3/4 of the last place (53 bits first, then the place of 2^-1074).
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda"


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    so = str(tmp_path_factory.mktemp("fft") / "libfft_probe.so")
    subprocess.run(["g++", "-O2", "-w", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(CUDA, "include"),
                    os.path.join(ROOT, "tests", "fft_probe.cpp"), "-o", so], check=True, capture_output=True)
    return ctypes.CDLL(so)


def _nearest(f, x0):
    """f 2^(x0 - 1022) exactly, in units of the last place of the double next to it."""
    from fractions import Fraction
    v = Fraction(int(f)) * Fraction(2) ** (int(x0) - 1022)
    e = max(v.__abs__().numerator.bit_length() - v.denominator.bit_length() - 1, -1022)
    if abs(v) >= Fraction(2) ** (e + 1):
        e += 1
    return v, Fraction(2) ** (e - 52)


@pytest.mark.parametrize("lo,hi", [(-62, 0), (-3, 8), (0, 100), (1900, 1960)])
def test_results_are_the_nearest_doubles(probe, lo, hi):
    from fractions import Fraction
    r = np.random.default_rng(hi)
    n = 4000
    f = r.integers(-2**61, 2**61, n) >> r.integers(0, 61, n)
    x0 = r.integers(lo, hi + 1, n).astype(np.int32)
    f[:4] = [0, 1, -1, 2**61]
    f = f.astype(np.int64)
    a, b = np.zeros(n), np.zeros(n)
    probe.fx_out(n, f.ctypes.data_as(ctypes.c_void_p), x0.ctypes.data_as(ctypes.c_void_p),
                 a.ctypes.data_as(ctypes.c_void_p), b.ctypes.data_as(ctypes.c_void_p))
    for i in range(n):
        v, ulp = _nearest(f[i], x0[i])
        for got in (a[i], b[i]):
            assert np.isfinite(got) and abs(Fraction(got) - v) <= ulp * Fraction(3 if abs(v) < Fraction(2)**-1022 else 2, 4)


@pytest.mark.parametrize("scale", [0.0, 5e-324, 1e-320, 1e-308, 1e-305, 1e-290, 1.0, 1e300])
@pytest.mark.parametrize("r1", [4, 8, 16])
def test_pencils_of_any_size(probe, r1, scale):
    r = np.random.default_rng(int(r1))
    v = r.standard_normal(2 * r1 * r1) * scale
    out = np.zeros_like(v)
    probe.fx_round_trip(len(v), v.ctypes.data_as(ctypes.c_void_p), r1.bit_length() - 1,
                        out.ctypes.data_as(ctypes.c_void_p))
    # 2^-55 of the largest component is cut off, then the nearest double (a multiple of 2^-1074)
    assert np.abs(out - v).max() <= 2.0**-52 * np.abs(v).max() + 2.0**-1074
