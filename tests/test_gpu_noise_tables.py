"""The FP64 normals are the same bits with and without the tables that the step reads
them from (there are none where 25 MB of device memory cannot be had)."""
import ctypes
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_tables_hold_what_the_kernels_form():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = os.path.join(HERE, "_build", "libnoise_tables_check.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-shared", "-o", tmp, os.path.join(HERE, "helpers", "noise_tables_check.cu")],
                   check=True)
    os.replace(tmp, out)
    f = ctypes.CDLL(out).noise_tables_differ
    f.restype = ctypes.c_longlong
    assert f() == 0
