"""The halo that a block of the column march stages from its neighbours, replayed
on the host over ragged grids: every address lies in the cells that the
neighbour publishes (a chunk of eight layers may begin before the neighbour's
first layer and end beyond the pyramid), and every layer before a marched one
is there."""
import ctypes
import os
import platform
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    cxx = shutil.which("g++")
    if nvcc is None or cxx is None:
        pytest.skip("no CUDA headers or host compiler")
    inc = os.path.join(os.path.dirname(os.path.realpath(nvcc)), "..", "include")
    out = os.path.join(HERE, "host", f"_libmarch_halo_host_{platform.machine()}_{os.getpid()}.so")
    subprocess.check_call([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", inc, "-o", out, "-x", "c++",
                           os.path.join(HERE, "host", "march_halo_host.cu")])
    yield ctypes.CDLL(out)
    os.remove(out)


# rows and layers of a chunk: the mixed trace, the FP64 trace, A1
@pytest.mark.parametrize("rows,chunk,sectors", [(21, 8, 1), (7, 8, 1), (7, 1, 0)])
def test_staged_halo_lies_in_the_neighbours_cells(lib, rows, chunk, sectors):
    rng = np.random.default_rng(11)
    grids = [((33, 33, 33), (0, 0, 0)), ((146, 35, 206), (0, 0, 0)), ((223, 49, 102), (0, 0, 51)), ((64, 64, 64), (32, 32, 32))]
    for _ in range(60):
        n = rng.integers(1, 120, 3)
        grids.append((tuple(n), tuple(rng.integers(0, n + 1))))
    staged = 0
    for n, v in grids:
        out = (ctypes.c_longlong * 3)()
        lib.oots_host_march_halo(*[int(m) for m in n], (ctypes.c_int * 3)(*[int(m) for m in v]), rows, chunk, sectors, out)
        assert (out[1], out[2]) == (0, 0), (n, v, list(out))
        staged += out[0]
    assert staged > 10 ** 6


def test_limit_on_the_halo_lies_above_the_limit_on_other_blocks(lib):
    """The handing warp alone gives up on other blocks: its CTA's own limit is a multiple of that limit for
    every limit that can be set, up to the largest (a product that overflowed gave up at the first test)."""
    lib.oots_host_march_ready_limit.restype = ctypes.c_longlong
    lib.oots_host_march_ready_limit.argtypes = [ctypes.c_longlong]
    top = 2 ** 63 - 1
    for s in [1, 2, 2000, 1 << 22, 1 << 40, 1 << 53, 1 << 59, 1 << 60, 1 << 62, top]:
        assert lib.oots_host_march_ready_limit(s) >= min(1024 * s, top), s
