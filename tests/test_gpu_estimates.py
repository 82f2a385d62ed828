"""Estimates after a frame that was abandoned: those of the frame before."""
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
