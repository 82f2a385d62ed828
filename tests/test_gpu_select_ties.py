"""glmb_select_top_static where the boundary bin of its first histogram
outgrows the list one block finishes (equal and nearly equal weights, large
caps), on both sides of the sizes where the grid takes the digits over, and its sums
where many small weights stand beside a large one."""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_gpu_select import _reference, select  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

LIST = 2048     # keys of the boundary bin that are listed


def _case(kind, n, rng):
    if kind == "bin":               # n - 100 keys within the boundary bin, the rest far above and below
        lw = -7.25 + 1e-4 * rng.random(n)
        lw[:50] = 0.0
        lw[50:100] = -40.0
        return rng.permutation(lw)
    if kind == "near":              # 2^-32 apart: the last digits decide
        return -7.25 + 2.0 ** -32 * rng.integers(0, 1 << 14, n)
    if kind == "equal":
        return np.full(n, -7.25)
    if kind == "steps":             # equal in all digits but the second
        return -1.0 + 2.0 ** -20 * rng.integers(0, 7, n)
    lw = 3.0 * rng.normal(size=n) - rng.exponential(4.0, n)
    lw[rng.random(n) < 0.3] = -np.inf
    return lw


@pytest.mark.parametrize("kind,n,h_max,tau", [
    ("bin", LIST + 99, 500, 1e-9), ("bin", LIST + 100, 500, 1e-9), ("bin", LIST + 101, 500, 1e-9),
    ("near", 8191, 100, 1e-9), ("near", 1 << 15, 9000, 1e-9), ("near", (1 << 15) + 1, 9000, 1e-30),
    ("equal", 1 << 13, 7, 1e-9), ("equal", (1 << 13) + 1, 7, 1e-9), ("near", 1 << 13, 4000, 1e-9), ("near", 40_000, 20_000, 0.9e-4), ("near", 8193, 8000, 1e-9), ("near", 155_649, 70_001, 1e-12),
    ("near", 1_000_003, 999_999, 1e-9), ("steps", 40_007, 20_001, 1e-9), ("steps", 1_000_003, 20_000, 1e-5),
    ("equal", 1_000_003, 20_000, 1e-9), ("equal", 1 << 22, 1, 1e-9), ("equal", (1 << 22) + 1, 5, 1e-9),
    ("smooth", 1_000_003, 400_001, 1e-12)])
def test_boundary_bins_beyond_the_list(select, kind, n, h_max, tau):  # noqa: F811
    lw = _case(kind, n, np.random.default_rng(n + h_max))
    idx, out = select(lw, h_max, tau)
    ridx, rout = _reference(lw, h_max, tau)
    assert np.array_equal(idx, ridx)
    tol = 8 * 2.0 ** -53 * max(1.0, float(np.max(np.abs(lw[ridx]))) if len(ridx) else 1.0) + 1e-14
    assert len(out) == len(rout) and (len(out) == 0 or np.max(np.abs(out - rout)) <= tol)


def test_ties_take_little_longer_than_other_weights(select):  # noqa: F811
    """A million children with equal weights: one more pass over them per
    digit.  Before the grid took those digits, 22 times the time."""
    import torch

    def best(lw):
        import paper_2512_06230_gb300 as glmb
        f = glmb.load().glmb_select_top_static
        x = torch.from_numpy(lw).cuda()
        idx = torch.zeros(20_000, dtype=torch.int64, device="cuda")
        out = torch.zeros(20_000, dtype=torch.float64, device="cuda")
        n = torch.zeros(1, dtype=torch.int32, device="cuda")
        s = torch.cuda.current_stream()
        times = []
        for _ in range(30):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            assert f(x.data_ptr(), len(lw), 20_000, 1e-9, idx.data_ptr(), out.data_ptr(), n.data_ptr(),
                     s.cuda_stream) == 0
            b.record()
            s.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    rng = np.random.default_rng(1)
    assert best(_case("equal", 1_000_000, rng)) < 5 * best(_case("smooth", 1_000_000, rng))


@pytest.mark.parametrize("tail", [-16.0, -24.5, -30.25, -41.3, -41.8, -44.0])
def test_a_million_small_weights_beside_a_large_one(select, tail):  # noqa: F811
    """The log-sum-exp is log(1 + (n - 1) e^tail): its sum is rounded to 2^-53
    by each of at most 32 additions on the way to the largest weight's
    partial, once over all and once over the kept (whose sum is the same), so
    the largest weight's result is off by at most 64 units of 2^-53."""
    n = 1_000_000
    lw = np.full(n, tail)
    lw[n // 3] = 0.0
    idx, out = select(lw, 1, 1e-30)
    assert list(idx) == [n // 3] and abs(out[0]) <= 2.0 ** -52      # alone after the second normalisation
    idx, out = select(lw, n, 1e-30)
    key = np.longdouble(np.rint(tail * 2.0 ** 32)) * np.longdouble(2.0) ** -32
    s = float(np.log1p((n - 1) * np.exp(key)))
    assert len(idx) == n
    assert abs(out[n // 3] + s) <= 64 * 2.0 ** -53
