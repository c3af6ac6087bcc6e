"""The D3Q19 noise transform's order of operations.  In 16-bit storage a sum
that rounds differently in the last FP32 bit now and then lands on the
neighbouring stored value, and the local noise amplifies it: a state of 300
steps then differs by 1e-4 and more.  So the order is part of the results, and
every version of the library has to keep it."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_d3q19_transform_keeps_its_order(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path / "libtoc.so")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-Xcompiler", "-ffp-contract=off", "-shared", "-I",
                    os.path.join(ROOT, "paper_1606_07801_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "csrc", "transform_order_check.cu"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.toc_d3q19_mismatches.argtypes = [ctypes.c_void_p, ctypes.c_int]
    z = np.random.default_rng(7).standard_normal((2000, 18)).astype(np.float32)
    assert lib.toc_d3q19_mismatches(z.ctypes.data, len(z)) == 0
