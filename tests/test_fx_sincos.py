"""Sine and cosine of csrc/fx_math.cuh near their zeros, compiled for the
host: the result keeps its relative precision there, as the FP64 library's
does (the reference is 60-digit decimal arithmetic)."""
from __future__ import annotations

import ctypes as C
import os
import subprocess
from decimal import Decimal as D
from decimal import getcontext

import numpy as np
import pytest

SRC = """
#include "fx_math.cuh"
using namespace glmb;
extern "C" void f_sc(const double* x, double* s, double* c, int n) { for (int i = 0; i < n; ++i) fx::sincos_turn(fx::turn(x[i]), s[i], c[i]); }
extern "C" void f_sum(const double* x, const double* h, double* s, double* c, int n) {
  for (int i = 0; i < n; ++i) fx::sincos_turn(fx::turn(x[i]) + fx::turn(h[i]), s[i], c[i]);
}
extern "C" int f_in(double x, double lim) { return fx::in_turn_range(x, lim) ? 1 : 0; }
"""
getcontext().prec = 70
PI = D("3.14159265358979323846264338327950288419716939937510582097494459230781640628620899862803")
TOL = D(2) ** -53 * (1 + D(2) ** -5)    # the result's rounding, and 2^-58 for argument and series


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxs")
    inc = os.path.join(os.path.dirname(__file__), "..", "paper_2512_06230_gb300", "csrc")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fsanitize=shift", "-fsanitize-undefined-trap-on-error",
                    "-I", inc, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _sin_cos(x):
    """Of a Decimal, by Taylor's series after taking whole quarter turns off."""
    n = int((x / (PI / 2)).to_integral_value())
    r = x - n * (PI / 2)
    s = t = r
    c = u = D(1)
    for k in range(1, 40):
        t *= -r * r / ((2 * k) * (2 * k + 1))
        u *= -r * r / ((2 * k - 1) * (2 * k))
        s += t
        c += u
    return [(s, c), (c, -s), (-s, -c), (-c, s)][n % 4]


def _arguments():
    rng = np.random.default_rng(7)
    x = [2.0 ** rng.uniform(-60, 0, 300) * rng.choice([-1, 1], 300), rng.uniform(-7, 7, 300),
         rng.uniform(-1e9, 1e9, 300), np.array([0.0, 2.0 ** -60, -2.0 ** -60, 1e-9, 0.5, 1.0, 64.0, 2.0 ** 29, -2.0 ** 29])]
    k = np.concatenate([np.arange(1, 40), rng.integers(1, 600_000_000, 200)])
    near = np.array([float(PI / 2 * int(m)) for m in k])      # the doubles nearest to the zeros
    x += [near, -near, np.nextafter(near, 0), near + 1e-9, near - 2.0 ** -40]
    return np.concatenate(x)


def _check(s, c, want):
    for a, b, (ws, wc) in zip(s, c, want):
        assert abs(D(float(a)) - ws) <= TOL * abs(ws), (a, ws)
        assert abs(D(float(b)) - wc) <= TOL * abs(wc), (b, wc)


def test_relative_precision_everywhere(lib):
    x = _arguments()
    s, c = np.empty_like(x), np.empty_like(x)
    lib.f_sc(_p(x), _p(s), _p(c), len(x))
    _check(s, c, [_sin_cos(D(float(v))) for v in x])


def test_sums_of_two_angles(lib):
    rng = np.random.default_rng(8)
    x = np.concatenate([rng.uniform(-7, 7, 200), 2.0 ** rng.uniform(-40, 0, 200), np.zeros(50)])
    h = np.concatenate([rng.uniform(-0.5, 0.5, 200), -x[200:400] * (1 + 2.0 ** -20), 2.0 ** rng.uniform(-59, -2, 50)])
    h = np.where(np.abs(h) < 0.5, h, h / 4)
    s, c = np.empty_like(x), np.empty_like(x)
    lib.f_sum(_p(x), _p(h), _p(s), _p(c), len(x))
    _check(s, c, [_sin_cos(D(float(a)) + D(float(b))) for a, b in zip(x, h)])


def test_range(lib):
    """What the fixed-point form takes: 0 and magnitudes from 2^-60 up to a limit."""
    lib.f_in.argtypes, lib.f_in.restype = [C.c_double, C.c_double], C.c_int
    for x, ok in [(0.0, 1), (-0.0, 1), (2.0 ** -60, 1), (-2.0 ** -60, 1), (np.nextafter(2.0 ** -60, 0), 0), (5e-324, 0),
                  (0.4999, 1), (0.5, 0), (-0.5, 0), (np.inf, 0), (-np.inf, 0), (np.nan, 0), (-np.nan, 0)]:
        assert lib.f_in(x, 0.5) == ok, x
