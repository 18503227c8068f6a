"""tab_all (value, difference and slope of ln P in one read) against the three
functions it stands for, on the host: columns below, in and beyond the table, on
its nodes and next to them, increments inside an interval, over a node, over
many intervals, past the end, and none.

Tolerance: the position t in an interval carries the rounding of ln N, at most
eps * 56 / (32.2 / 511) = 9e2 eps (2e-13 in FP64, 6e-5 in FP32), and the table's
slope changes by less than its own size over an interval, so values that take t
from ln(N + dN) or from t(N) + dt agree to 1e-11 and 1e-4 relative."""
import ctypes
import os
import platform
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SIG, T = 6.3e-18, 4.0e4


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    cxx = shutil.which("g++")
    if nvcc is None or cxx is None:
        pytest.skip("no CUDA headers or host compiler")
    inc = os.path.join(os.path.dirname(os.path.realpath(nvcc)), "..", "include")
    src = os.path.join(HERE, "host", "tab_all_host.cu")
    out = os.path.join(HERE, "host", f"_libtab_all_host_{platform.machine()}_{os.getpid()}.so")
    subprocess.check_call([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", inc, "-o", out, "-x", "c++", src, "-x", "none",
                           os.path.join(HERE, "..", "paper_1201_5651_gb300", "csrc", "tables.cpp")])
    L = ctypes.CDLL(out)
    d, v = ctypes.c_double, ctypes.c_void_p
    L.oots_host_tab_nodes.argtypes = [d, d, v]
    L.oots_host_tab_both.argtypes = [ctypes.c_int, d, d, v, v, ctypes.c_int, v]
    L.oots_host_tab_both.restype = None
    yield L
    os.remove(out)


@pytest.mark.parametrize("precision,tol", [(0, 1e-11), (1, 1e-4)])
def test_tab_all_matches_the_three_functions(lib, precision, tol):
    nodes = np.empty(4096)
    nodes = nodes[:lib.oots_host_tab_nodes(T, SIG, nodes.ctypes.data)]
    rng = np.random.default_rng(3)
    N = np.concatenate([[0.0, nodes[0] / 2, nodes[-1] * 2], nodes, np.nextafter(nodes, 0), np.nextafter(nodes, np.inf),
                        10.0 ** rng.uniform(9.0, 24.2, 2000)])
    f = np.concatenate([[0.0], 10.0 ** rng.uniform(-12, 4, 12), [nodes[1] / nodes[0] - 1.0, 1.0]])
    N, f = [a.ravel().copy() for a in np.meshgrid(N, f)]
    dN = N * f
    dN[N == 0.0] = 1e9
    out = np.empty((N.size, 6))
    lib.oots_host_tab_both(precision, T, SIG, N.ctypes.data, dN.ctypes.data, N.size, out.ctypes.data)
    got, want = out[:, :3], out[:, 3:]
    fin = np.isfinite(want)
    assert np.array_equal(got[~fin], want[~fin])
    assert np.all(np.abs(got[fin] - want[fin]) <= tol * np.abs(want[fin]))
