"""The FP64 Box-Muller pairs on the host, over all 2^24 arguments of each part.

The radius: -2 ln u0 is rounded to FP64 once (2^-53, halved by the square
root) from a value good to a quarter of that, and the square root is rounded
once: relative 2^-53 (0.5 + 0.125 + 1), with the second-order terms below 1.64
2^-53.  The angle: a base angle of one rounding and a small part of two
(half as large as the result at most, next to an axis, where the base is
exact on it and has one rounding of up to twice the result's size beside it),
and the rounding of their sum: relative 2^-53 (2 + 1 + 1), absolute 2^-53 (1 + 1)
and the small part's 2^-62.
"""
import ctypes
import os
import platform
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_errors_over_all_arguments(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double is FP64 here")
    out = str(tmp_path / "libbmc.so")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-Xcompiler", "-ffp-contract=off", "-shared", "-I",
                    os.path.join(ROOT, "paper_1606_07801_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "csrc", "bm64_check.cu"), "-o", out], check=True)
    e = np.zeros(5)
    ctypes.CDLL(out).bmc_errors(ctypes.c_void_p(e.ctypes.data))
    print(platform.machine(), "radius max %.3g rms %.3g, angle max %.3g rms %.3g, absolute %.3g" % tuple(e))
    assert e[0] <= 1.64 * 2.0**-53
    assert e[2] <= 4 * 2.0**-53
    assert e[4] <= 2.0**-52 * 1.01
