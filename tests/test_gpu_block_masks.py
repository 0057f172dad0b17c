"""The pixel-block masks of the list entries against lists without them.

Models of more than 2^24 Gaussians carry no masks (the key has no room beside the index): every
compositing warp then evaluates every entry of its tile at every pixel. The same Gaussians behind
2^24 others that are culled must give the same image, transmittance and contributor counts bit for
bit, whatever the splats' shapes, and the same gradient sums up to the order of their additions
(at most some 700 partial sums, one per pixel block, so 2 * 700 * 2^-24 of the sum of magnitudes)."""
import dataclasses
import math

import numpy as np
import pytest
import torch

from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, DeviceModel, Renderer

pytestmark = pytest.mark.gpu

N = 1500
FILL = 1 << 24


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


def shapes(kind):
    m = synth.make_model(61, N, 1, mask=0x7)
    g0 = m.g0.copy()
    st = synth.Stream(61, 70)
    if kind == "needles":  # up to some hundred times longer than wide, in every direction
        g0[7, :N] = math.log(0.01) + st.uniform(N) * math.log(100.0)
        g0[8:10, :N] = math.log(2e-4)
        g0[0:3, :N] *= 1.5  # some centred outside the frame
    elif kind == "faint":  # opacities around 1/255, where the reach shrinks to nothing
        g0[7:10, :N] += math.log(4.0)
        g0[10, :N] = -5.5 + 0.1 * st.normal(N)
    elif kind == "large":  # rectangles of many tiles (the cursor path of the scatter)
        g0[7:10, :N] += math.log(20.0)
        g0[10, :N] = -2.0
    return dataclasses.replace(m, g0=g0)


def behind(m, dev):
    """m's Gaussians at indices FILL ..., the others behind the near plane."""
    pad = FILL + m.n_pad
    g0 = torch.zeros(14, pad, device=dev)
    g0[2] = -5.0
    g0[3] = 1.0
    g0[:, FILL:] = torch.from_numpy(m.g0).to(dev)
    dg = torch.zeros(1, 3, pad, device=dev)
    dg[:, :, FILL:] = torch.from_numpy(m.dg).to(dev)
    return DeviceModel(FILL + m.n, 1, m.mask, g0, dg, torch.zeros_like(g0), torch.zeros_like(dg))


@pytest.mark.parametrize("kind", ["needles", "faint", "large", "plain"])
@pytest.mark.parametrize("tile,stage", [((16, 16), 64), ((8, 32), 128), ((16, 16), 256)])
def test_masked_lists_render_like_unmasked_ones(renderer, kind, tile, stage):
    m = shapes(kind)
    b = synth.make_batch([m], [synth.Frame(0, 173, 121)], seed=61, jitter_deg=10, random_bg=True)
    got = []
    for model in (None, [behind(m, "cuda:0")]):
        db = DeviceBatch(b, "cuda:0", tile=tile, smem_batch=stage, models=model)
        img, T, n = renderer.forward(db)
        renderer.backward(db, 1.0 + torch.arange(img.numel(), device="cuda:0") % 7, T, n)
        lay = renderer.layout(db)
        sums = renderer.ws[lay.grad2d: lay.grad2d + 48 * db.total_rec].view(torch.float32).view(-1, 12)
        got.append((img, T, n, sums[-m.n_pad:, :9].double()))
    renderer.ws = None
    (i0, T0, n0, s0), (i1, T1, n1, s1) = got
    assert int((n0 > 0).sum()) > 0
    assert torch.equal(i0, i1) and torch.equal(T0, T1) and torch.equal(n0, n1)
    assert float((s0[:, 6:] - s1[:, 6:]).abs().sub(1e-4 * s0[:, 6:]).max()) <= 0  # positive terms only
    assert bool(((s0 - s1).abs().amax(0) <= 1e-4 * s0.abs().amax(0)).all())
