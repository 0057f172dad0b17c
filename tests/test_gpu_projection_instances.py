"""The projection's instances by channel mask, frames per model, blendshape rows and binding: records, rectangles,
offsets and lists bit for bit against the oracle's, at the edges of the rules that choose one."""
import pytest

import oracle
from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import Renderer

from gpu_helpers import compare_decisions, read_intermediates, run_gpu_forward

pytestmark = pytest.mark.gpu

MASK_ALL = sum(1 << c for c in range(14) if c != 10)


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


def check(renderer, models, frames):
    batch = synth.make_batch(models, frames, seed=171, jitter_deg=10)
    r, db, _, _, _ = run_gpu_forward(batch, (16, 16), 64, renderer)
    stats = compare_decisions(batch, oracle.forward(batch, do_render=False), read_intermediates(r, db), db)
    assert stats["pairs"] > 0


# rows of blendshapes: 52, 65 and 832 of thirteen channels, 63 and 66 of three (64 is the edge)
@pytest.mark.parametrize("mask,k", [(MASK_ALL, 4), (MASK_ALL, 5), (MASK_ALL, 64), (0x7, 21), (0x7, 22)])
@pytest.mark.parametrize("nb", [1, 8, 9, 17])
def test_masks_read_at_run_time(renderer, nb, mask, k):
    models = [synth.make_model(171, 97, k, mask=mask), synth.make_model(172, 33, 3, mask=mask)]
    check(renderer, models, [synth.Frame(0, 96, 80)] * nb + [synth.Frame(1, 50, 60)])


@pytest.mark.parametrize("mask", [synth.MASK_MEAN_SCALE_COLOR, synth.MASK_PAPER, 0x7])
@pytest.mark.parametrize("nb", [8, 9, 17])
def test_bound_and_unbound_models(renderer, nb, mask):
    mesh = synth.make_head_mesh(8, 12, 24)
    models = [synth.make_bound_model(173, 130, 6, mesh, mask=mask), synth.make_model(174, 40, 3, mask=mask)]
    check(renderer, models, [synth.Frame(0, 96, 80, synth.frame_verts(mesh, 173, f)) for f in range(nb)] + [synth.Frame(1, 50, 60)])
