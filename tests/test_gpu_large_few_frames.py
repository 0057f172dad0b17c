"""The projection of large models rendered by few frames (from 20,000 Gaussians and up to four frames a thread reads
the blendshape rows itself, for one frame or for two): records, rectangles, offsets and lists bit for bit
against the oracle's, at Gaussian counts around the CTAs' 64, at blendshape counts around the unrolled four,
and with a small second model of fewer frames."""
import pytest

import oracle
from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import Renderer

from gpu_helpers import compare_decisions, read_intermediates, run_gpu_forward

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


def check(renderer, models, frames):
    batch = synth.make_batch(models, frames, seed=191, jitter_deg=10)
    r, db, _, _, _ = run_gpu_forward(batch, (16, 16), 64, renderer)
    assert compare_decisions(batch, oracle.forward(batch, do_render=False), read_intermediates(r, db), db)["pairs"] > 0


@pytest.mark.parametrize("mask", [synth.MASK_MEAN_SCALE_COLOR, synth.MASK_PAPER])
@pytest.mark.parametrize("nb", [1, 2, 3, 4])
@pytest.mark.parametrize("n,k", [(20000, 1), (20001, 4), (20033, 7), (20033, 13)])
def test_large_model_few_frames(renderer, n, k, nb, mask):
    models = [synth.make_model(191, n, k, mask=mask), synth.make_model(192, 70, max(1, k - 2), mask=mask)]
    check(renderer, models, [synth.Frame(0, 96, 80)] * nb + [synth.Frame(1, 50, 60)] * max(1, nb - 1))


@pytest.mark.parametrize("mask", [synth.MASK_MEAN_SCALE_COLOR, synth.MASK_PAPER])
@pytest.mark.parametrize("nb", [1, 3])
def test_large_bound_model_few_frames(renderer, nb, mask):
    mesh = synth.make_head_mesh(8, 12, 24)
    models = [synth.make_bound_model(193, 20030, 6, mesh, mask=mask), synth.make_model(194, 70, 5, mask=mask)]
    check(renderer, models, [synth.Frame(1, 50, 60)] + [synth.Frame(0, 96, 80, synth.frame_verts(mesh, 193, f)) for f in range(nb)])
