"""The allocation-free trace clears the march's counters itself: a call that another
one cut across, and that left them behind, does not reach the calls after it (the
march, handed a ticket past its last block, would write nothing and report success)."""
import ctypes
import os
import platform
import shutil
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_counters_start_at_zero():
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("no CUDA compiler")
    out = os.path.join(HERE, "device", f"_libnoalloc_counters_{platform.machine()}_{os.getpid()}.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-shared", "-Xcompiler",
                           "-fPIC", "-o", out, os.path.join(HERE, "device", "noalloc_counters.cu")])
    try:
        L = ctypes.CDLL(out)
        L.oots_test_noalloc_counters.restype = ctypes.c_longlong
        L.oots_test_noalloc_counters.argtypes = [ctypes.c_int, ctypes.c_uint, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
        for precision, dtype in ((0, torch.float64), (1, torch.float32)):
            x = torch.ones(20 ** 3, dtype=dtype, device="cuda")
            N = torch.empty_like(x)
            for left in (0, 1, 1 << 20):
                assert L.oots_test_noalloc_counters(precision, left, 20, x.data_ptr(), N.data_ptr()) == 0, left
    finally:
        os.remove(out)
