"""The FP32-pair regulator of the split epilogues (csrc/ff.cuh) on the CPU.

ff.cuh is compiled for the host (same operations in the same order; the GPU's
reciprocal seed is replaced by a division) and compared with FP64 on the
arguments the epilogues meet. Bounds: D is exact to 2^-48 of the operands, so
1/D and 1 - exp(-c D^2) are held to 2^-40 relative for |D| >= 1/4 and operands
up to about 9 (cancellation costs at most 2^6 of the 48 bits, squared).
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cmath>
#include "ff.cuh"
using namespace dsrg;
extern "C" void reg(const double* ca, const double* eb, double c, int n, double* inv, double* om,
                    double* sum) {
  ff tab[8];
  for (int m = 0; m < 8; ++m) tab[m] = ff_exp_entry(m);
  const ff k = ff_reg_scale(c);
  ff acc = {0.f, 0.f};
  for (int i = 0; i < n; ++i) {
    const ff D = ff_diff(ff_from(ca[i]), ff_from(eb[i]));
    const ff r = ff_inv(D), g = ff_one_minus_exp(D, k, tab);
    inv[i] = ff_to(r);
    om[i] = ff_to(g);
    ff_acc(acc, ff_mul(g, r));
  }
  *sum = ff_to(acc);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda = "/usr/local/cuda/include"
    if not gxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("ff")
    src, so = d / "ff.cpp", d / "libff.so"
    src.write_text(SRC)
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-std=c++17", "-I", cuda, "-I",
                    os.path.join(ROOT, "paper_1603_00561_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("c", [0.0, 1e-9, 1e-3, 0.1, 1.0, 2.0, 37.0])
def test_regulator_pairs(lib, c):
    r = np.random.default_rng(5)
    n = 100000
    ca = r.uniform(-4.0, -0.3, n) - r.uniform(0.05, 5.0, n)
    eb = r.uniform(-1.0, 5.0, n)
    ca[: n // 4] = eb[: n // 4] + r.choice([-1.0, 1.0], n // 4) * r.uniform(0.25, 0.5, n // 4)
    keep = np.abs(ca - eb) >= 0.25
    ca, eb = np.ascontiguousarray(ca[keep]), np.ascontiguousarray(eb[keep])
    n = ca.size
    inv, om, s = np.empty(n), np.empty(n), ctypes.c_double()
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.reg(p(ca), p(eb), ctypes.c_double(c), n, p(inv), p(om), ctypes.byref(s))
    D = ca - eb
    assert np.abs(inv * D - 1.0).max() < 2.0 ** -40
    ref = -np.expm1(-c * D * D)
    if c == 0.0:
        assert np.all(om == 0.0) and s.value == 0.0
    else:
        assert np.abs(om / ref - 1.0).max() < 2.0 ** -40
        assert abs(s.value / np.sum(ref / D) - 1.0) < 2.0 ** -40
