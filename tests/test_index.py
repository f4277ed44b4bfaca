"""Index arithmetic of the kernels (csrc/index.cuh) on the CPU, at sizes whose arrays are
larger than 2^32 elements."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "index.cuh"
extern "C" void split(const unsigned long long* r, int n, int nV, int* xu, int* e, int* f) {
  for (int i = 0; i < n; ++i) dsrg::split_xu_ef((size_t)r[i], nV, xu[i], e[i], f[i]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if not gxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("index")
    src, so = d / "index.cpp", d / "libindex.so"
    src.write_text(SRC)
    subprocess.run([gxx, "-O2", "-shared", "-fPIC", "-std=c++17", "-I", cuda, "-I",
                    os.path.join(ROOT, "paper_1603_00561_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("nV", [1, 3, 372, 46341, 65535, 65536, 65537, 66000, 130000])
def test_virtual_pair_positions(lib, nV):
    rng = np.random.default_rng(nV)
    n = 1000
    xu = rng.integers(0, 64, n)
    e, f = rng.integers(0, nV, n), rng.integers(0, nV, n)
    e[:4], f[:4] = [0, 0, nV - 1, nV - 1], [0, nV - 1, 0, nV - 1]
    r = (xu.astype(np.uint64) * np.uint64(nV) + e.astype(np.uint64)) * np.uint64(nV) + f.astype(np.uint64)
    got = [np.zeros(n, np.int32) for _ in range(3)]
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.split(p(r), n, nV, *(p(a) for a in got))
    for a, b in zip(got, (xu, e, f)):
        assert np.array_equal(a, b)
