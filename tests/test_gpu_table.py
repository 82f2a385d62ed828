"""The gated table (one kernel: prediction, gating, pieces of the pair arrays)
at the sizes where its split can go wrong: one to eight warps per component,
detection counts at and around the 32-bit words of its gate bits, one and many
components.  The table is compared with the gate restated in FP64 from the
components the library reports, and the frame graph's form (which predicts in
the table kernel) with the separate calls, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glmb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_06230_gb300 as g
    g.build()
    return g


def _frame(dim, n, M, seed):
    rng = np.random.default_rng(seed)
    extent = 400.0
    births = []
    for _ in range(n):
        A = rng.normal(size=(2 * dim, 2 * dim))
        births.append((0.6, np.concatenate([rng.uniform(0, extent, dim), rng.normal(size=dim)]),
                       np.diag([80.0] * dim + [9.0] * dim) + A @ A.T))
    Z = rng.uniform(0, extent, (M, dim))
    for i in range(M):
        if n and i % 3 == 0:
            Z[i] = births[i % n][1][:dim] + rng.normal(scale=12.0, size=dim)
    return births, Z.astype(np.float32)


def _cfg(dim, n, M):
    return dict(dim_x=2 * dim, dim_z=dim, dt=1.0, q=1.0, R=25.0 * np.eye(dim), p_s=0.99, p_d=0.9, lambda_d=1.0,
                clutter_rate=5.0, volume=400.0 ** dim, gate=18.4, h_max=4, h_up=4, tau=1e-6, seed=9, score_mode=0,
                max_tracks=n + 4, max_meas=max(M, 1), max_births=max(n, 1), max_pairs=max(64, n * M))


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n,M", [(1, 0), (1, 1), (1, 31), (1, 32), (3, 33), (5, 64), (2, 65), (9, 129), (1, 255),
                                 (7, 257), (4, 513), (1, 1025), (40, 2049), (700, 40)])
def test_table_against_the_gate_restated(glmb, dim, n, M):
    births, Z = _frame(dim, n, M, 100 * n + M)
    cfg = _cfg(dim, n, M)
    f, g = glmb.Filter(cfg), glmb.Filter(cfg)
    f.predict(births)
    f.update(Z)
    pairs, comps = f.pairs(), f.components()
    assert np.all(np.diff(pairs["ptr"].astype(np.int64)) >= 0) and pairs["ptr"][-1] == len(pairs["meas"])
    R = 25.0 * np.eye(dim)
    for c in range(n):
        # the frame's components are births (one frame from the empty GLMB),
        # so the reported mean and covariance are the ones the gate used
        m, P = comps["mean"][c][:dim], comps["cov"][c][:dim, :dim]
        S = P + R
        e = Z.astype(np.float64) - m
        d2 = np.einsum("ij,jk,ik->i", e, np.linalg.inv(S), e)
        lo, hi = int(pairs["ptr"][c]), int(pairs["ptr"][c + 1])
        got = pairs["meas"][lo:hi].astype(np.int64)
        assert np.all(np.diff(got) > 0)
        inside = np.zeros(M, bool)
        inside[got] = True
        clear = np.abs(d2 - 18.4) > 1e-5 * 18.4        # the parity contract's gate margin
        assert np.array_equal(inside[clear], (d2 <= 18.4)[clear])
        ref = np.log(0.9) - 0.5 * (d2[got] + np.linalg.slogdet(S)[1] + dim * np.log(2 * np.pi))
        assert np.allclose(pairs["logC"][lo:hi], ref, atol=5e-5, rtol=0)   # the contract's log C tolerance
        assert np.allclose(pairs["e"][lo:hi], e[got], atol=1e-4, rtol=2e-5)
    f.prune()
    g.step(births, Z)                                   # the frame graph
    q = g.pairs()
    for k in ("ptr", "meas", "logC", "q", "e"):
        assert np.array_equal(pairs[k], q[k]), k
    assert f.export_state() == g.export_state()
    f.close()
    g.close()
