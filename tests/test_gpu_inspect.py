"""The inspection calls of the pair table (pairs, gate features, logits and
usage), whose order is the table's (component, then detection) whatever place
the pairs took: after a frame whose pairs overflowed the table, and over
tables larger than the calls' work area."""
from __future__ import annotations

import ctypes as C

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
    births = [(0.6, np.concatenate([rng.uniform(0, 60, dim), rng.normal(size=dim)]),
               np.diag([30.0] * dim + [4.0] * dim)) for _ in range(n)]
    return births, rng.uniform(0, 60, (M, dim)).astype(np.float32)


def _cfg(dim, n, M, max_pairs, **kw):
    cfg = dict(dim_x=2 * dim, dim_z=dim, dt=1.0, q=1.0, R=9.0 * np.eye(dim), p_s=0.99, p_d=0.9, lambda_d=1.0,
               clutter_rate=5.0, volume=60.0 ** dim, gate=18.4, h_max=4, h_up=4, tau=1e-6, seed=9, score_mode=0,
               max_tracks=n + 4, max_meas=M, max_births=n, max_pairs=max_pairs)
    cfg.update(kw)
    return cfg


def _particle(cfg):
    out = dict(cfg, dim_x=5, model=1, n_particles=64, sigma_a=1.0, sigma_w=0.05, ess_frac=0.5, score_mode=1)
    return out


def _particle_births(births):
    return [(r, np.array([m[0], m[1], 3.0, 0.3, 0.01]), np.diag([30.0, 30.0, 1.0, 0.1, 0.01])) for r, m, _ in births]


@pytest.mark.parametrize("kind", ["2d", "3d", "particles"])
@pytest.mark.parametrize("frame", ["update", "step"])
@pytest.mark.parametrize("n,M", [(40, 33), (300, 70)])
def test_pairs_of_an_overflowed_frame(glmb, kind, frame, n, M):
    """The frame fails, and the table's first max_pairs pairs are still
    those of a filter with room for all."""
    dim = 3 if kind == "3d" else 2
    births, Z = _frame(dim, n, M, n + M)
    big = _cfg(dim, n, M, n * M)
    if kind == "particles":
        big, births = _particle(big), _particle_births(births)
    a = glmb.Filter(big)
    a.predict(births)
    a.update(Z)
    ref, comps = a.pairs(), a.components()
    K = len(ref["meas"])
    cap = K // 3
    assert cap > 50
    b = glmb.Filter(dict(big, max_pairs=cap))
    for _ in range(2):                     # the frame is refused, and refused again
        if frame == "update":
            b.predict(births)
            b.update(Z)
        else:
            with pytest.raises(glmb.GlmbError) as ei:
                b.step(births, Z)
            assert ei.value.status == 3
        got = b.pairs()
        assert len(got["meas"]) == cap and np.array_equal(got["ptr"], ref["ptr"])
        for k in ("meas", "logC", "q", "e"):
            assert np.array_equal(got[k], ref[k][:cap]), k
        whole = ref["ptr"][1:].astype(np.int64) <= cap      # components with all their pairs
        assert whole.any() and np.array_equal(b.components()["dprob"][whole], comps["dprob"][whole])
        if frame == "update":
            with pytest.raises(glmb.GlmbError) as ei:
                b.prune()
            assert ei.value.status == 3
    b.step(births, Z[:0])                  # a frame without detections runs
    a.close()
    b.close()


def test_capacity_is_checked_before_anything_is_built(glmb):
    births, Z = _frame(2, 40, 33, 5)
    f = glmb.Filter(_cfg(2, 40, 33, 40 * 33))
    f.step(births, Z)
    n, h = C.c_int64(), C.c_int()
    x = np.zeros(5, np.float32)
    p = x.ctypes.data_as(C.c_void_p)
    K = len(f.pairs()["meas"])
    assert f.lib.glmb_get_pairs(f.h, None, p, None, None, None, 1000, 1, C.byref(n)) == 3 and n.value == K
    assert f.lib.glmb_gate_features(f.h, p, 1, C.byref(n)) == 3 and n.value == K
    assert f.lib.glmb_gate_usage(f.h, p, 1, None, 0, C.byref(n), C.byref(h)) == 3 and n.value == K
    f.close()


@pytest.mark.parametrize("n,M", [(1, 1), (3, 200), (60, 300), (500, 90)])
def test_features_logits_and_usage_in_table_order(glmb, n, M):
    """More pairs than the hypotheses have room for: the calls take several
    rounds through their work area, and agree with the pairs."""
    from paper_2512_06230_gb300.gate import init_params, logits
    births, Z = _frame(2, n, M, 7 * n + M)
    f = glmb.Filter(_cfg(2, n, M, n * M, h_max=2, h_up=4, max_tracks=3 * n + 8))
    f.set_gate(init_params(1, np.zeros(5), np.full(5, 10.0)), 0.0, f.GATE_SCORE)
    f.step(births, Z)
    pr, comps = f.pairs(), f.components()
    K = len(pr["meas"])
    X, z = f.gate_features(), f.gate_logits()
    used, _ = f.gate_usage()
    assert len(X) == len(z) == len(used) == K
    comp = np.repeat(np.arange(n), np.diff(pr["ptr"].astype(np.int64)))
    if K:
        assert np.allclose(X[:, 1], np.linalg.norm(pr["e"], axis=1), rtol=1e-6)
        assert np.allclose(X[:, 4], comps["logdetS"][comp], rtol=0, atol=0)
        assert np.allclose(z, logits(init_params(1, np.zeros(5), np.full(5, 10.0)), X), rtol=0, atol=0)
    hyp = f.hypotheses()
    want = np.zeros(K, np.uint8)
    lab = {(int(a), int(b)): c for c, (a, b) in enumerate(zip(comps["label_k"], comps["label_b"]))}
    for j in range(len(hyp["logw"])):
        lo, hi = int(hyp["ptr"][j]), int(hyp["ptr"][j + 1])
        cs = [lab[int(a), int(b)] for a, b in zip(hyp["label_k"][lo:hi], hyp["label_b"][lo:hi])]
        for i, t in enumerate(hyp["theta"][j][:M]):
            if t:
                c = cs[int(t) - 1]
                a, b = int(pr["ptr"][c]), int(pr["ptr"][c + 1])
                want[a + int(np.nonzero(pr["meas"][a:b] == i)[0][0])] = 1
    assert np.array_equal(used, want)
    f.close()
