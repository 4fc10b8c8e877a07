"""The count of sampled steps of a call (flb_host.h), run on the host: the steps t
of [ta, tb) with t >= warmup and (t - warmup) % every == 0, for every schedule
that flb_set_sampling takes, up to the largest 64-bit ones."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
MAX = 2 ** 63 - 1


@pytest.fixture(scope="module")
def sampled():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = os.path.join(HERE, "_build", "libschedule_check.so")
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + f".tmp{os.getpid()}"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-shared", "-o", tmp, os.path.join(HERE, "helpers", "schedule_check.cu")],
                   check=True)
    os.replace(tmp, out)
    f = ctypes.CDLL(out).sampled
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_longlong] * 4
    return f


def test_small_schedules(sampled):
    for ta in range(0, 9):
        for tb in range(ta, 14):
            for warmup in range(0, 12):
                for every in range(0, 7):
                    want = sum(t >= warmup and (t - warmup) % every == 0 for t in range(ta, tb)) if every else 0
                    assert sampled(ta, tb, warmup, every) == want, (ta, tb, warmup, every)


@pytest.mark.parametrize("warmup", [0, 3, 10, 2 ** 40, MAX])
@pytest.mark.parametrize("every", [2 ** 31, 2 ** 62, MAX - 1, MAX])
def test_long_intervals(sampled, warmup, every):
    for ta, tb in ((0, 5), (5, 10), (10, 20), (2 ** 40, 2 ** 40 + 7), (2 ** 40 - 3, 2 ** 40 + 7)):
        want = sum(t >= warmup and (t - warmup) % every == 0 for t in range(ta, tb))
        assert sampled(ta, tb, warmup, every) == want, (ta, tb)
