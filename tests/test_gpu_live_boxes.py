"""Saturating blocks: the staged entries are cut to the pixels still in the walk, in stages of 64 entries for
batches of few tiles and of 32 otherwise. Lists without block masks (models of more than 2^24 Gaussians) are not cut:
the same Gaussians must give the same image, transmittance and contributor counts bit for bit, and the same gradient
sums up to the order of their additions (at most some 100 partial sums of 16 pixels, one per half block: 2 * 100 *
2^-24 of the sum of magnitudes, and colour sums have positive terms only)."""
import dataclasses
import math

import pytest
import torch

from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer

from test_gpu_block_masks import behind

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("opacity", [-2.0, 3.0])
@pytest.mark.parametrize("sizes,tile", [([(64, 48)], (16, 16)), ([(64, 48), (512, 512)], (16, 16)), ([(50, 61)], (8, 32)),
                                        ([(50, 61), (520, 520)], (8, 32))])
def test_cut_entries_change_nothing(renderer, sizes, tile, opacity):
    n = 6000
    m = synth.make_model(111, n, 1, mask=0x7)
    g0 = m.g0.copy()
    g0[7:10, :n] += math.log(2.0)
    g0[10, :n] = opacity + 0.5 * synth.Stream(111, 70).normal(n)
    m = dataclasses.replace(m, g0=g0)
    b = synth.make_batch([m], [synth.Frame(0, w, h) for w, h in sizes], seed=111, jitter_deg=10, random_bg=True)
    got = []
    for model in (None, [behind(m, "cuda:0")]):
        db = DeviceBatch(b, "cuda:0", tile=tile, models=model)
        img, T, k = renderer.forward(db)
        renderer.backward(db, 1.0 + torch.arange(img.numel(), device="cuda:0") % 7, T, k)
        lay = renderer.layout(db)
        sums = renderer.ws[lay.grad2d: lay.grad2d + 48 * db.total_rec].view(torch.float32).view(-1, 12)
        at = db.rec_offsets[0] + db.models[0].n_pad - m.n_pad
        got.append((img, T, k, sums[at: at + m.n_pad, :9].double()))
    renderer.ws = None
    (i0, T0, n0, s0), (i1, T1, n1, s1) = got
    assert int((n0 > 0).sum()) > 0
    if opacity > 0:
        assert float(T0[: sizes[0][0] * sizes[0][1]].min()) < 1e-3  # blocks do saturate
    assert torch.equal(i0, i1) and torch.equal(T0, T1) and torch.equal(n0, n1)
    assert float((s0[:, 6:] - s1[:, 6:]).abs().sub(1e-4 * s0[:, 6:]).max()) <= 0
    assert bool(((s0 - s1).abs().amax(0) <= 1e-4 * s0.abs().amax(0)).all())
