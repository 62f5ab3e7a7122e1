"""Division by a fixed divisor (csrc/fast_div.cuh), built for the host, where it runs the same
multiplication and shift as on the device: equal to the integer division for every numerator
below 2^31 that lies next to a multiple of the divisor, and at the ends of the range."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("fast_div") / "libfast_div_host.so")
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_0901_3163_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fast_div_host.cu"), "-o", out], check=True, capture_output=True)
    L = ctypes.CDLL(out)
    L.fast_div_first_wrong.argtypes = [ctypes.c_uint, ctypes.c_void_p, ctypes.c_int]
    return L


def test_quotients(lib):
    top = 2**31 - 1
    rng = np.random.default_rng(0)
    divisors = list(range(1, 700)) + [2**k + e for k in range(10, 31) for e in (-1, 0, 1)]
    divisors += [top, top - 1] + [int(x) for x in rng.integers(700, top, 400)]
    for d in divisors:
        q = np.unique(np.concatenate([np.arange(64), rng.integers(0, top // d + 1, 500), [top // d]]))
        n = np.concatenate([q * d + e for e in (-1, 0, 1)] + [[0, 1, top - 1, top]])
        n = np.ascontiguousarray(n[(n >= 0) & (n <= top)], dtype=np.int32)
        bad = lib.fast_div_first_wrong(d, n.ctypes.data, len(n))
        assert bad < 0, (d, n[bad])
