"""The thread-per-child draw at the sizes where its mapping can go wrong: few
and many draws per parent (one CTA then spans many parents, whose records may
not fit in shared memory), counts that do not divide the CTA, and small CTAs.
Children, retained sets and states equal the warp-per-child draw's exactly."""
from __future__ import annotations

import pytest

from tests.test_gpu_paths import _run_lockstep, glmb  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("preset,h_up", [("tiny", 1), ("tiny", 7), ("tiny", 129), ("mid", 33), ("sweep_N50", 100),
                                         ("sweep_N50", 31), ("sweep_N50", 3)])
def test_thread_draw_equals_warp_draw(glmb, preset, h_up):  # noqa: F811
    F = glmb.Filter
    over = dict(max_meas=400, max_births=16, max_tracks=300) if preset == "mid" else {}
    _run_lockstep(glmb, preset, 21, 8, [F.OPT_DRAW_WARP, F.OPT_DRAW_THREAD], h_up=h_up, **over)
