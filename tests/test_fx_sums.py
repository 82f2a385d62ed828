"""Sums of exponentials in fixed point (csrc/fx_math.cuh), compiled for the
host with shifts checked: small terms keep their own precision beside a large
one, and no shift reaches the width of its operand."""
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
extern "C" void f_one(const unsigned long long* d, double* y, double* z, int n) {
  for (int i = 0; i < n; ++i) {
    fx::ExpSum s;
    s.add(d[i], T.exp2);
    y[i] = s.value();
    z[i] = fx::exp_fixed(d[i], T.exp2);
  }
}
extern "C" double f_sum(const unsigned long long* d, int n) {
  fx::ExpSum s;
  for (int i = 0; i < n; ++i) s.add(d[i], T.exp2);
  return s.value();
}
"""
LD = np.longdouble
if np.finfo(LD).nmant < 63:
    pytest.skip("no extended precision here", allow_module_level=True)
ONE = 1 << 32


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxsum")
    inc = os.path.join(os.path.dirname(__file__), "..", "paper_2512_06230_gb300", "csrc")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fsanitize=shift", "-fsanitize-undefined-trap-on-error",
                    "-I", inc, str(src), "-o", str(so)], check=True)
    out = C.CDLL(str(so))
    out.f_sum.restype = C.c_double
    return out


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _exp(d):
    return np.exp(-(d.astype(LD) / LD(ONE)))


def test_each_value(lib):
    rng = np.random.default_rng(2)
    d = np.concatenate([rng.integers(0, 90 * ONE, 5000), (ONE * rng.exponential(2.0, 2000)).astype(np.int64),
                        np.arange(0, 129 * ONE, ONE // 2), [0, 1, 2, 41 * ONE, 42 * ONE - 1, 42 * ONE, 63 * ONE - 1, 63 * ONE,
                        int(41.59 * ONE), (1 << 39) - 1, 1 << 39, 1 << 62, (1 << 63) - 1]]).astype(np.uint64)
    y, z = np.empty(len(d)), np.empty(len(d))
    lib.f_one(_p(d), _p(y), _p(z), len(d))
    want = _exp(d)
    # the result's rounding and 2^-54 of the series, argument and table
    near = d < (1 << 39)
    assert np.all(np.abs(z[near].astype(LD) / want[near] - 1) <= 2.0 ** -53 + 2.0 ** -54)
    assert np.all(z[~near] == 0.0)
    # in units of 2^-90, truncated; nothing below one
    assert np.all(np.abs(y.astype(LD) - want) <= (2.0 ** -53 + 2.0 ** -54) * want + LD(2) ** -89.8)


@pytest.mark.parametrize("tail", [0.0, 1e-9, 5.5, 16.0, 30.25, 41.6, 41.99, 42.0, 60.0])
def test_sums_of_small_terms(lib, tail):
    d = np.full(31, int(tail * ONE), np.uint64)
    s = lib.f_sum(_p(d), 31)
    want = 31 * _exp(d[:1])[0]
    assert abs(LD(s) - want) <= (2.0 ** -53 + 2.0 ** -54) * want + 31 * LD(2) ** -90
    d[0] = 0
    s = lib.f_sum(_p(d), 31)
    assert abs(LD(s) - (1 + 30 * _exp(d[1:2])[0])) <= 2.0 ** -53 * s
