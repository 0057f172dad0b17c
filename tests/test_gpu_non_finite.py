"""Infinite and undefined values stay with the pixels and Gaussians they belong to. A Gaussian whose
colour is not finite changes only the pixels that blend it, whatever else its splat was staged for."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


def batch_of(n=2000, colours=None):
    """One avatar in a frame whose blocks hold all of a pixel's cases; colours: {Gaussian: RGB}."""
    m = synth.make_model(141, n, 3, mask=0x7)
    g0 = m.g0.copy()
    g0[11:14, :n] = 0.5
    for i, c in (colours or {}).items():
        g0[11:14, i] = c
    return synth.make_batch([dataclasses.replace(m, g0=g0)], [synth.Frame(0, 173, 121)], seed=141, jitter_deg=10,
                            random_bg=True)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("tile,stage", [((16, 16), 64), ((8, 32), 64), ((16, 16), 256)])
def test_a_colour_reaches_only_the_pixels_that_blend_it(renderer, tile, stage, value):
    odd = range(0, 2000, 40)

    def render(c):
        db = DeviceBatch(batch_of(colours={i: c for i in odd}), "cuda:0", tile=tile, smem_batch=stage)
        img, T, n = renderer.forward(db)
        return img.view(3, 121, 173), T, n

    plain, T0, n0 = render(0.5)
    far, _, _ = render(1e6)  # a blended alpha is at least 1/255: 1e6 moves every pixel that blends one
    got, T, n = render(value)
    blends = (far != plain).any(0)
    assert 100 < int(blends.sum()) < blends.numel() - 100
    assert torch.equal(T, T0) and torch.equal(n, n0)
    assert torch.equal(got[:, ~blends], plain[:, ~blends])
    assert not bool(torch.isfinite(got[:, blends]).any())
