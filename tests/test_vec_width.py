"""Sites per thread of the register-pull step kernels, on the host: a vector of that many values lies on a
multiple of its size in both buffers whatever their addresses, divides Lx, and is as wide as on aligned buffers
where the addresses allow."""
import ctypes
import itertools
import os
import shutil
import subprocess

import pytest

import paper_1606_07801_gb300 as lb

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BYTES = {lb.F32: 4, lb.F64: 8, lb.F32_F16: 2, lb.F32_BF16: 2}


def test_width_follows_the_buffers(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path / "libvwc.so")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-shared", "-I",
                    os.path.join(ROOT, "paper_1606_07801_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "csrc", "vec_width_check.cu"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.vwc_width.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_ulonglong,
                              ctypes.c_ulonglong, ctypes.c_int]
    base = 1 << 20
    for lat, prec in itertools.product((lb.D1Q3, lb.D2Q9, lb.D3Q19, lb.D2Q5), BYTES):
        b = BYTES[prec]
        for lx, sites in itertools.product((1, 2, 3, 4, 6, 8, 12, 1023, 1024), (2048, 1 << 17, 1 << 19, 1 << 24)):
            best = lib.vwc_width(lat, prec, lx, sites, base, base, b)
            assert best in (1, 2, 4) and lx % best == 0
            for i, j in itertools.product(range(5), range(5)):
                vx = lib.vwc_width(lat, prec, lx, sites, base + i * b, base + j * b, b)
                assert lx % vx == 0 and (base + i * b) % (vx * b) == 0 and (base + j * b) % (vx * b) == 0
                allowed = max(v for v in (1, 2, 4) if i % v == 0 and j % v == 0)
                assert vx == min(best, allowed)
