"""The work memory that operators keep between calls (csrc/device_memory.cpp), built for the host
against a stand-in for the CUDA allocator: how much is kept, that an allocation that does not fit
gets the idle buffers of every operator before it fails, and that calls of several host threads
never hold the same buffer."""
import ctypes
import os
import shutil
import subprocess
import threading

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20
OOM = -8


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are not available")
    out = str(tmp_path_factory.mktemp("memory") / "libdevice_memory_host.so")
    csrc = os.path.join(ROOT, "paper_0901_3163_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", csrc,
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"),
                    os.path.join(csrc, "device_memory.cpp"), os.path.join(ROOT, "tests", "device_memory_host.cpp"),
                    "-o", out, "-pthread"], check=True, capture_output=True)
    L = ctypes.CDLL(out)
    vp, sz, ip = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
    for name, res, args in (("dm_limit", None, [sz]), ("dm_used", sz, []), ("dm_pool_new", vp, []),
                            ("dm_pool_delete", None, [vp]), ("dm_take", vp, [vp, sz, ctypes.POINTER(ip)]),
                            ("dm_bytes", sz, [vp]), ("dm_give", None, [vp, vp]), ("dm_alloc", ip, [sz]),
                            ("dm_hammer", ip, [vp, sz, ip, ip])):
        f = getattr(L, name)
        f.restype, f.argtypes = res, args
    return L


@pytest.fixture
def pools(lib):
    lib.dm_limit(64 << 30)
    made = [lib.dm_pool_new() for _ in range(12)]
    yield made
    for p in made:
        lib.dm_pool_delete(p)
    assert lib.dm_used() == 0


def _take(lib, pool, nbytes):
    rc = ctypes.c_int(0)
    return lib.dm_take(pool, nbytes, ctypes.byref(rc)), rc.value


def _keep(lib, pool, sizes):
    bufs = [_take(lib, pool, s)[0] for s in sizes]
    for b in bufs:
        lib.dm_give(pool, b)


def test_kept_and_reused(lib, pools):
    _keep(lib, pools[0], [10 * MB, 64 * MB, 65 * MB])
    assert lib.dm_used() == 74 * MB                      # the 65 MB one is freed at once
    b, _ = _take(lib, pools[0], 5 * MB)
    assert lib.dm_bytes(b) == 10 * MB and lib.dm_used() == 74 * MB
    lib.dm_give(pools[0], b)
    _keep(lib, pools[0], [20 * MB, 30 * MB, 40 * MB, 50 * MB, 60 * MB])
    # four at most: the largest ones stay (20 MB took the 64 MB buffer)
    assert lib.dm_used() <= 4 * 64 * MB
    lib.dm_pool_delete(pools.pop(0))
    assert lib.dm_used() == 0


def test_an_allocation_gets_the_idle_buffers(lib, pools):
    for p in pools[:3]:
        _keep(lib, p, [60 * MB])
    lib.dm_limit(lib.dm_used() + 10 * MB)
    assert lib.dm_alloc(100 * MB) == 0                   # any allocation of the library
    assert lib.dm_used() == 0
    for p in pools[:3]:
        _keep(lib, p, [60 * MB])
    b, rc = _take(lib, pools[0], 150 * MB)               # one for a call's work memory
    assert b and rc == 0
    lib.dm_give(pools[0], b)
    held, _ = _take(lib, pools[1], 60 * MB)              # in use: never taken away
    b, rc = _take(lib, pools[0], 150 * MB)
    assert not b and rc == OOM
    assert lib.dm_bytes(held) == 60 * MB
    lib.dm_give(pools[1], held)


def test_bound_over_all_operators(lib, pools):
    for p in pools:
        _keep(lib, p, [60 * MB] * 4)
    assert lib.dm_used() <= 512 * MB
    for p in pools:                                      # still usable
        b, rc = _take(lib, p, 60 * MB)
        assert b and rc == 0
        lib.dm_give(p, b)


def test_threads(lib, pools):
    got = []
    ts = [threading.Thread(target=lambda m=m: got.append(lib.dm_hammer(pools[m % 2], 3 * MB, 4000, m + 1)))
          for m in range(6)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert got == [0] * 6
