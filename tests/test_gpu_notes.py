"""The notes of the thread-per-child draw: a filter that never draws so does
not hold them, and one that cannot have them runs without, with the same
results (its noted children are redone by the warp kernel)."""
from __future__ import annotations

import pytest

import scenes

pytestmark = pytest.mark.gpu

NOTE = 64   # bytes per child slot


@pytest.fixture(scope="module")
def glmb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_06230_gb300 as g
    g.build()
    return g


class Allocator:
    """torch's caching allocator; refuses blocks of `refuse` bytes."""

    def __init__(self, refuse=None):
        self.refuse, self.sizes, self.live = refuse, [], {}

    def alloc(self, nbytes):
        import torch
        self.sizes.append(nbytes)
        if nbytes == self.refuse:
            return None
        p = torch.cuda.caching_allocator_alloc(nbytes)
        self.live[p] = nbytes
        return p

    def free(self, p):
        import torch
        del self.live[p]
        torch.cuda.caching_allocator_delete(p)


@pytest.mark.parametrize("preset,force", [("tiny", False), ("tiny", True), ("mid", False)])
def test_with_and_without_the_notes(glmb, preset, force):
    sc = scenes.make_scene(scenes.preset(preset), 31)
    cfg = sc.filter_config()
    size = NOTE * cfg["h_max"] * cfg["h_up"]
    ref, al, no = glmb.Filter(cfg), Allocator(), Allocator(refuse=size)
    f, g = (glmb.Filter(cfg, allocator=(x.alloc, x.free)) for x in (al, no))
    assert (size in al.sizes) == (preset == "mid")
    if force:
        for x in (ref, f, g):
            x.set_launch_options(glmb.Filter.OPT_DRAW_THREAD)
    redone = 0
    for fr in sc.frames[:14]:
        for x in (ref, f, g):
            x.step(fr.births, fr.Z)
        assert f.info()["n_draw_overflow"] <= g.info()["n_draw_overflow"]
        redone += g.info()["n_draw_overflow"]
        assert ref.export_state() == f.export_state() == g.export_state()
    assert (size in al.sizes) == (preset == "mid" or force)
    assert (redone > 0) == (preset == "mid" or force)
    ref.close()
    f.close()
    g.close()
    assert not al.live and not no.live
