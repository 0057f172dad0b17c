"""Infinite and undefined values stay with the pixels and Gaussians they belong to. A Gaussian whose
colour is not finite changes only the pixels that blend it, whatever else its splat was staged for; a pixel whose
dL/dimg is not finite makes the sums of the Gaussians that it blends undefined, and no others'."""
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


def batch_of(n=2000, colours=None, sizes=((173, 121),)):
    """One avatar in a frame whose blocks hold all of a pixel's cases, and in others; colours: {Gaussian: RGB}."""
    m = synth.make_model(141, n, 3, mask=0x7)
    g0 = m.g0.copy()
    g0[11:14, :n] = 0.5
    for i, c in (colours or {}).items():
        g0[11:14, i] = c
    return synth.make_batch([dataclasses.replace(m, g0=g0)], [synth.Frame(0, w, h) for w, h in sizes], seed=141,
                            jitter_deg=10, random_bg=True)


# alone: few tiles, stages of 64 entries; with the second frame stages of 32
SIZES = [((173, 121),), ((173, 121), (512, 520))]


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("tile,stage", [((16, 16), 64), ((8, 32), 64), ((16, 16), 256)])
@pytest.mark.parametrize("sizes", SIZES)
def test_a_colour_reaches_only_the_pixels_that_blend_it(renderer, sizes, tile, stage, value):
    odd = range(0, 2000, 40)

    def render(c):
        db = DeviceBatch(batch_of(colours={i: c for i in odd}, sizes=sizes), "cuda:0", tile=tile, smem_batch=stage)
        img, T, n = renderer.forward(db)
        return db.image_views(img)[0], T, n

    plain, T0, n0 = render(0.5)
    far, _, _ = render(1e6)  # a blended alpha is at least 1/255: 1e6 moves every pixel that blends one
    got, T, n = render(value)
    blends = (far != plain).any(0)
    assert 100 < int(blends.sum()) < blends.numel() - 100
    assert torch.equal(T, T0) and torch.equal(n, n0)
    assert torch.equal(got[:, ~blends], plain[:, ~blends])
    assert not bool(torch.isfinite(got[:, blends]).any())


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("channels", [(0,), (0, 1, 2)])
@pytest.mark.parametrize("tile", [(16, 16), (8, 32)])
@pytest.mark.parametrize("n", [2000, 30000])
@pytest.mark.parametrize("sizes", SIZES)
def test_a_pixel_gradient_reaches_only_what_the_pixel_blends(renderer, sizes, n, tile, channels, value):
    """n: blocks of a few entries, and of several stages. The other Gaussians' sums equal those with 0 at these pixels,
    up to the order of their additions (at most some 100 partial sums, one per half block, of which
    the nine sums' magnitudes add: 2 * 100 * 2^-24 of the largest, times ten)."""
    batch = batch_of(n, sizes=sizes)
    db = DeviceBatch(batch, "cuda:0", tile=tile)
    img, T, k = renderer.forward(db)
    ys, xs = torch.meshgrid(torch.arange(5, 121, 23, device="cuda:0"), torch.arange(3, 173, 19, device="cuda:0"), indexing="ij")
    bad = torch.zeros(121, 173, dtype=torch.bool, device="cuda:0")
    bad[ys, xs] = True
    clean = 1.0 + (torch.arange(3 * 121 * 173, device="cuda:0") % 7).view(3, 121, 173)

    def sums(dl):
        full = torch.ones_like(img)
        db.image_views(full)[0].copy_(dl)
        renderer.backward(db, full, T, k)
        lay = renderer.layout(db)
        return renderer.ws[lay.grad2d: lay.grad2d + 48 * db.total_rec].view(torch.float32).view(-1, 12)[:n, :9].clone()

    owned = sums(bad.float().expand(3, -1, -1))[:, 6] > 0  # w times 1: what the pixels blend
    assert 20 < int(owned.sum()) < n - 20
    odd, ref = clean.clone(), clean.clone()
    for c in range(3):
        ref[c][bad] = 0.0
        odd[c][bad] = value if c in channels else 0.0
    got, want = sums(odd), sums(ref)
    assert bool(torch.isfinite(got[~owned]).all()) and int((want[~owned] != 0).sum()) > 0
    assert bool(((got - want)[~owned].abs() <= 1e-4 * want.abs().amax(0)).all())
    for c in range(3):  # the channels whose gradient is finite keep their colour sums
        if c in channels:
            assert not bool(torch.isfinite(got[owned, 6 + c]).any())
        else:
            assert bool(((got - want)[:, 6 + c].abs() <= 1e-4 * want[:, 6 + c].abs().max()).all())
