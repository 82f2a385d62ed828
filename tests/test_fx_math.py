"""The integer-arithmetic functions of the particle kernels (csrc/fx_math.cuh),
compiled for the host, against 64-bit-mantissa arithmetic: rounding of the
result (2^-53 relative) plus the argument's or the series' (2^-54 or less)."""
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
extern "C" void f_exp(const double* x, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = fx::exp_neg(x[i], T.exp2); }
extern "C" void f_log(const unsigned* w, double* y, double* r, int n) {
  for (int i = 0; i < n; ++i) {
    const fx::Val v = fx::neg2_log_unit(w[i], T.nlog, T.inv);
    y[i] = fx::to_double(v);
    r[i] = fx::to_double(fx::root(v));
  }
}
extern "C" void f_cos(const unsigned* w, double* y, int n) {
  for (int i = 0; i < n; ++i) {
    bool neg;
    const double v = fx::to_double(fx::cos_turn(w[i], neg));
    y[i] = neg ? -v : v;
  }
}
extern "C" void f_norm(const unsigned* w, const unsigned* u, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = fx::normal(w[i], u[i], T.nlog, T.inv); }
extern "C" void f_sc(const double* x, double* s, double* c, int n) { for (int i = 0; i < n; ++i) fx::sincos_turn(fx::turn(x[i]), s[i], c[i]); }
extern "C" void f_sinc(const double* x, double* y, int n) { for (int i = 0; i < n; ++i) y[i] = fx::sinc(x[i]); }
"""
LD = np.longdouble
if np.finfo(LD).nmant < 63:
    pytest.skip("no extended precision here", allow_module_level=True)
PI = LD(3141592653589793238) / LD(10) ** 18 + LD(4626433832795029) / LD(10) ** 34
TOL = 2.0 ** -53 + 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    inc = os.path.join(os.path.dirname(__file__), "..", "paper_2512_06230_gb300", "csrc")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", inc, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _words():
    rng = np.random.default_rng(3)
    w = rng.integers(0, 1 << 32, 4000, dtype=np.uint64).astype(np.uint32)
    edge = [0, 1, 2, 0x7FFFFFFF, 0x80000000, 0xFFFFFFFF, 0xFFFFFFFE, 0xFE000000 - 1, 0xFE000000, 0xFE000000 + 1,
            0xFDFFFFFF, 0x1FFFFFFF, 0x20000000, 0x3FFFFFFF, 0x40000000, 0x5FFFFFFF, 0x60000000, 0xC0000000]
    small = (w[:500] >> (np.arange(500, dtype=np.uint32) % 32)).astype(np.uint32)
    return np.concatenate([w, np.array(edge, np.uint32), small, ~small])


def test_exp(lib):
    rng = np.random.default_rng(4)
    x = np.concatenate([rng.uniform(0, 1, 1000), rng.uniform(0, 40, 1000), rng.uniform(0, 707.9, 1000),
                        2.0 ** rng.uniform(-300, 0, 500), [5e-324, 1e-310, np.log(2), 707.999, 708.0, 800.0, np.inf]])
    y = np.empty_like(x)
    lib.f_exp(_p(x), _p(y), len(x))
    want = np.exp(-x.astype(LD))
    ok = x < 708
    assert np.all(np.abs(y[ok].astype(LD) / want[ok] - 1) <= TOL)
    assert np.all(y[~ok] == 0.0)


def test_log(lib):
    w = _words()
    y, r = np.empty(len(w)), np.empty(len(w))
    lib.f_log(_p(w), _p(y), _p(r), len(w))
    d = (LD(2) ** 33 - (LD(2) * w.astype(LD) + 1)) / LD(2) ** 33   # 1 - u, exact
    want = -2 * np.log1p(-d)
    assert np.all(np.abs(y.astype(LD) / want - 1) <= TOL)
    assert np.all(np.abs(r.astype(LD) / np.sqrt(want) - 1) <= TOL)


def test_normal(lib):
    w = _words()
    u = np.roll(w, 17)
    y = np.empty(len(w))
    lib.f_norm(_p(w), _p(u), _p(y), len(w))
    d = (LD(2) ** 33 - (LD(2) * w.astype(LD) + 1)) / LD(2) ** 33
    size, c = np.sqrt(-2 * np.log1p(-d)), np.cos(2 * PI * ((LD(2) * u.astype(LD) + 1) / LD(2) ** 33))
    assert np.all(np.abs(y.astype(LD) - size * c) <= TOL * size * np.maximum(np.abs(c), LD(2) ** -8))


def test_cos_of_a_turn(lib):
    w = _words()
    y = np.empty(len(w))
    lib.f_cos(_p(w), _p(y), len(w))
    want = np.cos(2 * PI * ((LD(2) * w.astype(LD) + 1) / LD(2) ** 33))
    assert np.all(np.abs(y.astype(LD) - want) <= TOL * np.maximum(np.abs(want), LD(2) ** -8))


def test_sincos(lib):
    rng = np.random.default_rng(5)
    x = np.concatenate([rng.uniform(-7, 7, 2000), rng.uniform(-1e3, 1e3, 1000), 2.0 ** rng.uniform(-80, 0, 500),
                        np.pi / 4 * np.arange(-16, 17), [0.0, -0.0, 1e-300]])
    s, c = np.empty_like(x), np.empty_like(x)
    lib.f_sc(_p(x), _p(s), _p(c), len(x))
    assert np.all(np.abs(s.astype(LD) - np.sin(x.astype(LD))) <= TOL)
    assert np.all(np.abs(c.astype(LD) - np.cos(x.astype(LD))) <= TOL)


def test_sinc(lib):
    rng = np.random.default_rng(6)
    x = np.concatenate([rng.uniform(-0.4999, 0.4999, 2000), 2.0 ** rng.uniform(-200, -2, 500), [0.0, -0.0, 0.49999999]])
    y = np.empty_like(x)
    lib.f_sinc(_p(x), _p(y), len(x))
    xl = x.astype(LD)
    want = np.where(np.abs(xl) < 1e-12, LD(1), np.sin(xl) / np.where(xl == 0, LD(1), xl))
    assert np.all(np.abs(y.astype(LD) / want - 1) <= TOL)
