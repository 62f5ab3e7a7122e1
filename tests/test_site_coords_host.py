"""Coordinates of a site and of a checkerboard site by the multiplications and shifts that device
code uses (csrc/fast_div.cuh, dlz_internal.cuh, wilson_eo_site.cuh), built for the host: equal to
the integer divisions on ragged lattices, with extents of 1, and at the end of the largest ones."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("coords") / "libsite_coords_host.so")
    subprocess.run([nvcc, "-x", "cu", "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(ROOT, "paper_0901_3163_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "site_coords_host.cu"), "-o", out], check=True, capture_output=True)
    L = ctypes.CDLL(out)
    L.coords_first_wrong.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    L.eo_first_wrong.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return L


@pytest.mark.parametrize("dims", [(1, 1, 1, 7), (3, 5, 7, 9), (2, 3, 1, 4), (12, 10, 14, 18), (16, 16, 16, 32),
                                  (31, 33, 17, 8)])
def test_sites(lib, dims):
    d = (ctypes.c_int * 4)(*dims)
    assert lib.coords_first_wrong(d, 0, dims[0] * dims[1] * dims[2] * dims[3]) == -1


@pytest.mark.parametrize("dims", [(112, 112, 112, 127), (3, 5, 7, 1700000), (1, 9999, 1, 17000)])
def test_last_sites_of_large_lattices(lib, dims):
    d = (ctypes.c_int * 4)(*dims)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    assert V > 2**27 and 12 * V < 2**31
    assert lib.coords_first_wrong(d, V - 100000, 100000) == -1


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 6, 10, 2), (14, 2, 6, 8), (8, 8, 8, 16)])
@pytest.mark.parametrize("par", [0, 1])
def test_checkerboard(lib, dims, par):
    assert lib.eo_first_wrong((ctypes.c_int * 4)(*dims), par) == -1
