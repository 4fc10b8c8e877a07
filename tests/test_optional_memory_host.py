"""Device memory that a handle can do without (the mailboxes of cut lattices) is asked for
with what it needs and left out where only that can be had (flb_host.h, run on the host
with an allocator of limited memory)."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("free,need,extra,want", [
    (100, 80, 20, (100, True)), (99, 80, 20, (80, False)), (80, 80, 20, (80, False)), (79, 80, 20, None),
    (79, 80, 0, None), (80, 80, 0, (80, True))])
def test_extra_memory(free, need, extra, want):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = os.path.join(HERE, "_build", "liboptional_memory_check.so")
    src = os.path.join(HERE, "helpers", "schedule_check.cu")
    hdr = os.path.join(HERE, "..", "paper_1204_6734_gb300", "csrc", "flb_host.h")
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(hdr)):
        os.makedirs(os.path.dirname(out), exist_ok=True)
        tmp = out + f".tmp{os.getpid()}"
        subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                        "--expt-relaxed-constexpr", "-shared", "-o", tmp, src], check=True)
        os.replace(tmp, out)
    f = ctypes.CDLL(out).extra
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_longlong] * 3 + [ctypes.POINTER(ctypes.c_int)]
    got = ctypes.c_int(7)
    n = f(free, need, extra, ctypes.byref(got))
    assert ((n, bool(got.value)) if n >= 0 else None) == want
