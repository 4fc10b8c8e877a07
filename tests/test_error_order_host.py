"""Which error of a launch of many steps is kept (flb_kernels.cuh, run on the host): the
earliest one and, in its step, the lowest node; an earlier launch's stays. Step counters
are 32 bits and may wrap inside a launch."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def precedes():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = os.path.join(HERE, "_build", "liberror_order_check.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-shared", "-o", tmp, os.path.join(HERE, "helpers", "schedule_check.cu")],
                   check=True)
    os.replace(tmp, out)
    f = ctypes.CDLL(out).precedes
    f.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_uint, ctypes.c_uint,
                  ctypes.c_int]
    return lambda *a: bool(f(*a))


@pytest.mark.parametrize("t0", [0, 1000, 2 ** 31 - 3, 2 ** 32 - 5])
def test_order(precedes, t0):
    n, m = 10, 2 ** 32
    for a in range(n):
        for b in range(n):
            for na, nb in ((7, 7), (7, 9), (9, 7), (-1, 7), (7, -1)):
                assert precedes(1, na, (t0 + a) % m, nb, (t0 + b) % m, t0, n) == ((b, nb) < (a, na))
    assert precedes(0, 0, 0, 5, (t0 + 9) % m, t0, n)                      # nothing recorded yet
    for before in (1, 5, 2 ** 20, 2 ** 31):                               # an earlier launch's
        assert not precedes(1, 7, (t0 - before) % m, 5, t0, t0, n)
