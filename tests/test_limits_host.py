"""Kernel limits shared by all contexts of a process (csrc/limits.cpp), on the CPU with
a stand-in for the CUDA runtime: serving slots run one context per thread, with operators
of different sizes, and several devices may be in use.

Every thread must find at least the shared memory it asked for however the others'
calls fall; every device gets its own limit; a refused size changes nothing.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda"


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    so = str(tmp_path_factory.mktemp("limits") / "liblimits_probe.so")
    # -Bsymbolic: the stand-in, not a CUDA runtime that another test has loaded
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", os.path.join(CUDA, "include"),
                    os.path.join(ROOT, "tests", "limits_probe.cpp"),
                    os.path.join(ROOT, "paper_2003_11679_gb300", "csrc", "limits.cpp"), "-o", so, "-lpthread"],
                   check=True, capture_output=True)
    return ctypes.CDLL(so)


def test_threads_keep_what_they_asked_for(probe):
    assert probe.limits_race(20000) == 0


def test_each_device_has_its_own(probe):
    out = (ctypes.c_int * 4)()
    probe.limits_devices(out)
    assert list(out) == [100000, 100000, 1, -1]


def test_refused_sizes_change_nothing(probe):
    out = (ctypes.c_int * 2)()
    assert probe.limits_refused(out) == 0
    assert list(out) == [-1, 70000]


def test_no_kernel_sets_its_limits_elsewhere():
    csrc = os.path.join(ROOT, "paper_2003_11679_gb300", "csrc")
    for f in os.listdir(csrc):
        if f != "limits.cpp":
            assert "cudaFuncSetAttribute" not in open(os.path.join(csrc, f)).read(), f
