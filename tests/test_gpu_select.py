"""glmb_select_top_static against a NumPy restatement (stable sort by
fixed-point key, ties to the lower index) at the sizes where its passes can go
wrong: one child, block edges, ties that outgrow the boundary list, caps below
and above the candidates, no valid child, the one-pass and the
histogram-per-digit forms."""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def select():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_06230_gb300 as glmb
    glmb.build()
    f = glmb.load().glmb_select_top_static
    f.argtypes = [C.c_void_p, C.c_int64, C.c_int32, C.c_double, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    f.restype = C.c_int

    def run(lw, h_max, tau):
        x = torch.from_numpy(np.ascontiguousarray(lw, np.float64)).cuda()
        idx = torch.full((h_max,), -1, dtype=torch.int64, device="cuda")
        out = torch.zeros(h_max, dtype=torch.float64, device="cuda")
        n = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        s = torch.cuda.current_stream()
        assert f(x.data_ptr(), len(lw), h_max, tau, idx.data_ptr(), out.data_ptr(), n.data_ptr(), s.cuda_stream) == 0
        s.synchronize()
        k = int(n.item())
        return idx[:k].cpu().numpy(), out[:k].cpu().numpy()

    return run


def _reference(lw, h_max, tau):
    ok = np.nonzero(np.isfinite(lw) & (np.abs(lw) < 2.0 ** 30))[0]
    if not len(ok):
        return ok, np.zeros(0)
    key = np.rint(lw[ok] * 2.0 ** 32).astype(np.int64)
    x = (key - key.max()).astype(np.longdouble) * np.longdouble(2.0) ** -32
    lse = float(np.longdouble(key.max()) * np.longdouble(2.0) ** -32 + np.log(np.sum(np.exp(x))))
    at = key >= math.ceil((lse + math.log(tau)) * 2.0 ** 32)
    ok, key = ok[at], key[at]
    order = np.lexsort((ok, -key))[:h_max]
    keep = np.sort(order)
    if not len(keep):
        return ok[keep], np.zeros(0)
    x = (key[keep] - key.max()).astype(np.longdouble) * np.longdouble(2.0) ** -32
    return ok[keep], (x - np.log(np.sum(np.exp(x)))).astype(np.float64)


def _case(kind, n, rng):
    if kind == "ties":              # a few distinct values: a boundary bin far larger than the list
        return rng.integers(-3, 1, n).astype(np.float64)
    if kind == "equal":
        return np.full(n, -7.25)
    if kind == "none":
        return np.where(np.arange(n) % 3 == 0, np.nan, np.where(np.arange(n) % 3 == 1, -np.inf, 2.0 ** 31))
    lw = 3.0 * rng.normal(size=n) - rng.exponential(4.0, n)
    lw[rng.random(n) < 0.3] = -np.inf
    if kind == "huge":              # spans the whole range of valid log-weights
        lw *= 1e7
    return lw


@pytest.mark.parametrize("kind,n,h_max,tau", [
    ("mixed", 1, 1, 1e-5), ("mixed", 31, 5, 1e-5), ("mixed", 1024, 100, 1e-9), ("mixed", 1025, 2000, 1e-9),
    ("mixed", 100_003, 1, 1e-5), ("mixed", 100_003, 5000, 1e-9), ("mixed", 1_000_000, 20000, 1e-9),
    ("mixed", (1 << 22) + 1, 20000, 1e-9), ("ties", 50_000, 777, 1e-9), ("ties", 300_001, 100_000, 1e-9),
    ("equal", 4096, 1000, 1e-9), ("equal", 70_000, 70_000, 1e-9), ("huge", 20_000, 50, 1e-5),
    ("mixed", 5000, 5000, 1.0), ("mixed", 5000, 64, 0.5), ("none", 1000, 10, 1e-5)])
def test_selection_against_numpy(select, kind, n, h_max, tau):
    lw = _case(kind, n, np.random.default_rng(n + h_max))
    idx, out = select(lw, h_max, tau)
    ridx, rout = _reference(lw, h_max, tau)
    assert np.array_equal(idx, ridx)
    # a kept log-weight is a difference of values of magnitude |lse| and
    # |lse_kept|, each rounded to 2^-53 of it, over keys that are exact
    tol = 8 * 2.0 ** -53 * max(1.0, float(np.max(np.abs(lw[ridx]))) if len(ridx) else 1.0) + 1e-14
    assert len(out) == len(rout) and (len(out) == 0 or np.max(np.abs(out - rout)) <= tol)
