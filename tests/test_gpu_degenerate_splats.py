"""Splats far larger than any frame, up to those whose conic underflows to 0 (which reach no pixel), in lists
with pixel-block masks and in lists without them (models of more than 2^24 Gaussians): both give the same
bits."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer

from test_gpu_block_masks import behind

pytestmark = pytest.mark.gpu

N, GIANTS = 1500, 40


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("tile", [(16, 16), (8, 32)])
@pytest.mark.parametrize("log_scale", [(1, 4), (5, 9), (10, 14), (15, 17), (18, 24)])
def test_giants_with_and_without_masks(renderer, log_scale, tile):
    m = synth.make_model(151, N, 1, mask=0x7)
    g0 = m.g0.copy()
    lo, hi = log_scale
    u = synth.Stream(151, 70).uniform(3 * GIANTS).reshape(3, GIANTS)
    # the conic underflows for the largest ones, which are round: others of their size have no finite covariance
    g0[7:10, :GIANTS] = lo + (hi - lo) * (u[0] if lo >= 18 else u)
    g0[10, :GIANTS] = -3.0
    m = dataclasses.replace(m, g0=g0)
    b = synth.make_batch([m], [synth.Frame(0, 173, 121)], seed=151, jitter_deg=10, random_bg=True)
    got = []
    for model in (None, [behind(m, "cuda:0")]):
        db = DeviceBatch(b, "cuda:0", tile=tile, models=model)
        got.append(renderer.forward(db))
        lay = renderer.layout(db)
        at = db.total_rec - m.n_pad
        rect = renderer.ws[lay.rects: lay.rects + 8 * db.total_rec].cpu().numpy().view(np.uint16).reshape(-1, 4)[at: at + GIANTS]
        conic = renderer.ws[lay.records: lay.records + 48 * db.total_rec].view(torch.float32).view(-1, 12)[at: at + GIANTS, 2].cpu()
        kept = (rect[:, 2] > rect[:, 0]) & (rect[:, 3] > rect[:, 1])
        assert kept.sum() >= 10 and (int((conic[torch.from_numpy(kept)] == 0).sum()) > 0) == (lo >= 18)
    renderer.ws = None
    for x, y in zip(*got):
        assert torch.equal(x, y)
