"""Estimates where their handling can go wrong: after a frame that was
abandoned, at result blocks around 48 KB (where the launch's shared memory
passes the default limit only with the kernel's static part), and where the
estimates' kernel cannot be launched at all."""
from __future__ import annotations

import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glmb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_06230_gb300 as g
    g.build()
    return g


def _same(a, b):
    return a["n"] == b["n"] and all(np.array_equal(a[k], b[k]) for k in ("labels", "r", "mean", "cov", "pmf"))


@pytest.mark.parametrize("how", ["step", "enqueue", "batch"])
def test_abandoned_frame_keeps_the_estimates(glmb, how):
    """No clutter and a detection far from every track: no child has a weight,
    the frame fails, and the estimates stay those of the frame before."""
    sc = scenes.make_scene(scenes.preset("tiny"), 1004)
    far = np.array([[-5.0e4, -5.0e4]], np.float32)
    f = glmb.Filter(sc.filter_config())
    g = glmb.Filter(sc.filter_config(clutter_rate=0.0))
    for fr in sc.frames[:6]:
        f.step(fr.births, fr.Z)
    g.import_state(f.export_state())
    g.step([], far[:0])                     # a frame without detections
    before, state = g.estimates(), g.export_state()
    assert before["n"] > 0
    with pytest.raises(glmb.GlmbError) as ei:
        if how == "step":
            g.step([], far)
        elif how == "enqueue":
            g.step_enqueue([], far)
            g.step_finish()
        else:
            glmb.step_batch([g], [([], far)])
    assert ei.value.status == 5
    assert g.export_state() == state
    assert _same(g.estimates(), before)
    f.close()
    g.close()


def _small(max_tracks, **kw):
    rng = np.random.default_rng(11)
    births = [(0.7, np.concatenate([rng.uniform(0, 100, 2), rng.normal(size=2)]), np.diag([9.0, 9.0, 1.0, 1.0]))
              for _ in range(6)]
    Z = np.array([b[1][:2] for b in births[:5]], np.float32)
    cfg = dict(dim_x=4, dim_z=2, dt=1.0, q=1.0, R=4.0 * np.eye(2), p_s=0.99, p_d=0.9, lambda_d=1.0, clutter_rate=2.0,
               volume=1e4, gate=18.4, h_max=4, h_up=8, tau=1e-6, seed=3, score_mode=0, max_tracks=max_tracks,
               max_meas=64, max_births=8, max_components=256, max_pairs=4096)
    cfg.update(kw)
    return cfg, births, Z


@pytest.mark.parametrize("max_tracks", [511, 512, 4095, 4096, 6045, 6046, 6100, 6143, 6144, 6200, 20000])
def test_result_blocks_of_every_size(glmb, max_tracks):
    cfg, births, Z = _small(max_tracks)
    ref, f = glmb.Filter(_small(64)[0]), glmb.Filter(cfg)
    for k in range(3):
        for x in (ref, f):
            x.step(births if k == 0 else [], Z)
        a, b = ref.estimates(pmf_cap=65), f.estimates(pmf_cap=65)
        assert a["n"] > 0 and _same(a, b)
    ref.close()
    f.close()


def test_frame_whose_estimates_cannot_be_launched(glmb):
    """More tracks than a block can count in shared memory: each step reports
    the refused launch and leaves the state, and frames without the estimates
    run."""
    cfg, births, Z = _small(40000)
    f, ref = glmb.Filter(cfg), glmb.Filter(_small(64)[0])
    frame = f.info()["frame"]
    for _ in range(3):
        with pytest.raises(glmb.GlmbError) as ei:
            f.step(births, Z)
        assert ei.value.status == 4          # GLMB_E_CUDA
        info = f.info()
        assert info["frame"] == frame and info["n_graph_captures"] == 0 and info["n_graph_launches"] == 0
    f.set_step_estimates(False)
    for k in range(2):
        f.step(births if k == 0 else [], Z)
        ref.step(births if k == 0 else [], Z)
    assert f.export_state() == ref.export_state()
    f.close()
    ref.close()
