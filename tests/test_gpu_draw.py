"""The thread-per-child draw at the sizes where its mapping can go wrong: few
and many draws per parent (one CTA then spans many parents, whose records may
not fit in shared memory), counts that do not divide the CTA, and small CTAs.
Children, retained sets and states equal the warp-per-child draw's exactly."""
from __future__ import annotations

import pytest

import scenes

from tests.test_gpu_paths import _run_lockstep, glmb  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("preset,h_up", [("tiny", 1), ("tiny", 7), ("tiny", 129), ("mid", 33), ("sweep_N50", 100),
                                         ("sweep_N50", 31), ("sweep_N50", 3)])
def test_thread_draw_equals_warp_draw(glmb, preset, h_up):  # noqa: F811
    F = glmb.Filter
    over = dict(max_meas=400, max_births=16, max_tracks=300) if preset == "mid" else {}
    _run_lockstep(glmb, preset, 21, 8, [F.OPT_DRAW_WARP, F.OPT_DRAW_THREAD], h_up=h_up, **over)


@pytest.mark.parametrize("preset,frames", [("sweep_N1000", 3), ("sweep_N50", 9)])
def test_staging_threads_do_not_change_the_children(glmb, preset, frames):  # noqa: F811
    """Few large parents (1024 staging threads by default) and many small ones
    (64) against 32 and 128 threads."""
    sc = scenes.make_scene(scenes.preset(preset), 22)
    fs = []
    for threads in (0, 32, 128):
        f = glmb.Filter(sc.filter_config(max_births=1016, max_tracks=3200, max_meas=4200))
        f.set_tuning(stage_threads=threads)
        fs.append(f)
    for k, fr in enumerate(sc.frames[:frames]):
        for f in fs:
            f.predict(fr.births)
            f.update(fr.Z)
            f.prune()
        ref = fs[0].export_state()
        assert all(f.export_state() == ref for f in fs[1:]), k
