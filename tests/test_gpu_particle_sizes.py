"""One frame with the particle model against the FP64 oracle at the particle
counts where the update's blocks change: one, two and four particles to a
thread, remainders, and the particles in memory from 1025 on."""
from __future__ import annotations

import pytest

import scenes
from tests.test_gpu_particle import _cfg, _frame, glmb  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_,h_max", [(63, 100), (65, 100), (65, 300), (129, 100), (256, 100), (257, 100), (257, 300),
                                       (512, 100), (513, 100), (1025, 100)])
def test_particle_counts_at_the_block_sizes(oracle_mod, glmb, np_, h_max):  # noqa: F811
    p = scenes.CtrvParams(n_objects=5, frames=12, h_max=h_max, n_particles=np_, ess_frac=0.7)
    _frame(oracle_mod, glmb, _cfg(p, 504), scenes.ctrv_scene(p, 504), 8)
