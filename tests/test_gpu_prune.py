"""The in-frame selection at the sizes where its split changes: one block
alone, with its keys held or read again, and the cluster; the tau cut or the
cap binding.  The retained children are the unique ones at or above tau, the
h_max heaviest of them (ties by index), in index order."""
from __future__ import annotations

import numpy as np
import pytest

import scenes
from tests.test_gpu_paths import glmb  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("preset,h_max,h_up,over", [
    ("tiny", 5, 100, {}),            # one block, keys held, cap binds
    ("tiny", 40, 100, {}),           # one block, at most 4000 children
    ("tiny", 100, 150, {}),          # one block, keys read again
    ("tiny", 20, 823, {}),           # past one block's children by a few
    ("tiny", 4, 5000, {}),           # duplicate marking with one table
    ("tiny", 4, 1500, {}),           # tables of 48 KB
    ("sweep_N50", 60, 100, {}),      # 3-D, cap binds
    ("sweep_N50", 400, 331, {}),     # cluster, keys read again, cap binds
    ("sweep_N50", 3000, 100, {}),    # cluster, the cap does not bind at first
])
def test_retained_set(glmb, preset, h_max, h_up, over):  # noqa: F811
    sc = scenes.make_scene(scenes.preset(preset), 31)
    cfg = sc.filter_config(h_max=h_max, h_up=h_up, **over)
    f = glmb.Filter(cfg)
    for k, fr in enumerate(sc.frames[:9]):
        f.predict(fr.births)
        f.update(fr.Z)
        c = f.children()
        f.prune()
        idx, logw = f.retained()
        ok = np.flatnonzero(c["status"] == 1)
        w = c["logw"][ok]
        lse = w.max() + np.log(np.sum(np.exp(w - w.max())))
        cut = lse + np.log(cfg["tau"])
        # the sum's FP32 exponentials move the cut by about 1e-7
        sure, maybe = ok[w >= cut + 1e-6], ok[w >= cut - 1e-6]
        if len(sure) == len(maybe):
            want = np.sort(sure[np.lexsort((sure, -c["logw"][sure]))[:h_max]])
            assert np.array_equal(idx, want), k
            kept = c["logw"][want]
            kept = kept - (kept.max() + np.log(np.sum(np.exp(kept - kept.max()))))
            np.testing.assert_allclose(logw, kept, rtol=0, atol=1e-6)
