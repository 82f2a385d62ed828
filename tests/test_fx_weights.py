"""exp of a log-weight difference (csrc/fx_math.cuh), compiled for the host,
over the whole range of the FP64 library's function: subnormal results too."""
from __future__ import annotations

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

SRC = """
#include "fx_math.cuh"
using namespace glmb;
static constexpr fx::Tables T{};
extern "C" void f_w(const double* x, double* y, double* z, int n) {
  for (int i = 0; i < n; ++i) {
    y[i] = fx::exp_weight(x[i], T.exp2);
    z[i] = std::exp(x[i]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxw")
    inc = os.path.join(os.path.dirname(__file__), "..", "paper_2512_06230_gb300", "csrc")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", inc, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def test_every_range(lib):
    rng = np.random.default_rng(9)
    x = np.concatenate([-rng.uniform(0, 800, 4000), -rng.uniform(700, 750, 2000), rng.uniform(0, 1e-10, 50),
                        [0.0, -0.0, -5e-324, 5e-324, -707.999, -708.0, np.nextafter(-708.0, 0), np.nextafter(-708.0, -1e3),
                         -709.0, -744.0, -745.1, -745.14, -745.9, -746.0, -1e300, -np.inf, np.nan, -np.nan, 1e-16, 3.0]])
    y, z = np.empty_like(x), np.empty_like(x)
    p = [a.ctypes.data_as(C.c_void_p) for a in (x, y, z)]
    lib.f_w(*p, len(x))
    nan = np.isnan(x)
    assert np.all(np.isnan(y[nan]))
    x, y, z = x[~nan], y[~nan], z[~nan]
    # both are within an ulp of the exact value; 2^-1074 apart where subnormal
    assert np.all(np.abs(y - z) <= 2.0 ** -52 * z)
    low = x <= -708.0
    assert np.array_equal(y[low], z[low]) and np.any((y[low] > 0) & (y[low] < 2.0 ** -1022))
