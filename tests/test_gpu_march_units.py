"""The mixed march's reciprocal, square root and column sum against 64 bits, over the
values they meet (1 .. 1e6; square roots of 1 .. 3): the first two within 0.51 units in
the last place (a Newton step squares the approximation's error, a few units, and adds
one rounding of half a unit), the float-float sum exact to 2^-46 of the larger term
whichever of the two it is."""
import ctypes
import os
import platform
import shutil
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("no CUDA compiler")
    out = os.path.join(HERE, "device", f"_libmarch_units_{platform.machine()}_{os.getpid()}.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                           "-fPIC", "-o", out, os.path.join(HERE, "device", "march_units.cu")])
    L = ctypes.CDLL(out)
    L.oots_test_march_units.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3
    yield L
    os.remove(out)


@pytest.mark.parametrize("top", [3.0, 1e6])
def test_units_against_64_bits(lib, top):
    m = 1 << 20
    rng = np.random.default_rng(4)
    a = np.exp(rng.uniform(0.0, np.log(top), m)).astype(np.float32)
    b = (a * 10.0 ** rng.uniform(-6, 6, m)).astype(np.float32)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.empty(4, m, device="cuda")
    assert lib.oots_test_march_units(m, da.data_ptr(), db.data_ptr(), out.data_ptr()) == 0
    rcp, root, hi, lo = out.double().cpu().numpy()
    a, b = a.astype(np.float64), b.astype(np.float64)
    for got, want in ((rcp, 1 / a), (root, np.sqrt(a))):
        ulp = np.spacing(want.astype(np.float32)).astype(np.float64)
        assert float(np.max(np.abs(got - want) / ulp)) <= 0.51
    assert float(np.max(np.abs((hi - a - b) + lo) / np.maximum(a, b))) <= 2.0 ** -46
