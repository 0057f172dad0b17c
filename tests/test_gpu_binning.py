"""Projection and binning at the edges of their rules: models rendered by few frames (one thread per
Gaussian and frame pair) and by more (staged rows), Gaussian counts around the CTAs' pieces, blendshape counts
around the unrolled four, and frames at and past the tiles that a CTA counts in shared memory. Records,
rectangles, offsets and lists bit for bit against the oracle's."""
import dataclasses
import math

import pytest
import torch

import oracle
from paper_2503_12886_gb300 import api, synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer, stream_ptr

from gpu_helpers import compare_decisions, read_intermediates, run_gpu_forward

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


def check(renderer, batch, tile):
    r, db, _, _, _ = run_gpu_forward(batch, tile, 64, renderer)
    inter = read_intermediates(r, db)
    return compare_decisions(batch, oracle.forward(batch, tile=tile, do_render=False), inter, db, tile)


@pytest.mark.parametrize("mask", [synth.MASK_MEAN_SCALE_COLOR, synth.MASK_PAPER, 0x7])
@pytest.mark.parametrize("nb,n,k", [(1, 63, 1), (1, 65, 4), (2, 64, 5), (3, 257, 3), (4, 255, 8), (5, 256, 6)])
def test_few_frames(renderer, mask, nb, n, k):
    models = [synth.make_model(101, n, k, mask=mask), synth.make_model(102, 40, 7, mask=mask)]
    batch = synth.make_batch(models, [synth.Frame(0, 96, 80)] * nb + [synth.Frame(1, 50, 60)], seed=101, jitter_deg=10)
    assert check(renderer, batch, (16, 16))["pairs"] > 0


@pytest.mark.parametrize("tile", [(16, 16), (8, 32)])
@pytest.mark.parametrize("size", [(1536, 2048), (1552, 2048), (2049, 1999)])
def test_large_frames(renderer, tile, size):
    m = synth.make_model(103, 300, 3)
    g0 = m.g0.copy()
    g0[7:10, :20] += math.log(8.0)  # some rectangles of hundreds of tiles
    batch = synth.make_batch([dataclasses.replace(m, g0=g0)], [synth.Frame(0, *size), synth.Frame(0, 64, 48)], seed=103,
                             jitter_deg=10)
    assert check(renderer, batch, tile)["pairs"] > 0


@pytest.mark.parametrize("sizes", [[(1024, 1024)], [(1024, 1024), (16, 16)], [(16, 16)], [(1, 1)], [(1024, 1008), (250, 10)]])
def test_scan_by_one_cta(renderer, sizes):
    """Up to 4,096 tiles are scanned by one CTA: 4,096, 4,097, 1, 1 and 4,048 tiles."""
    m = synth.make_model(104, 3000, 3)
    batch = synth.make_batch([m], [synth.Frame(0, w, h) for w, h in sizes], seed=104, jitter_deg=10)
    assert check(renderer, batch, (16, 16))["pairs"] > 0


@pytest.mark.parametrize("sizes", [[(200, 150)], [(1024, 1024), (64, 48)], [(2049, 1999)]])
def test_binning_again_gives_the_same_lists(renderer, sizes):
    """rgba_bin_sort may run any number of times on one rgba_preprocess."""
    m = synth.make_model(105, 2000, 3)
    batch = synth.make_batch([m], [synth.Frame(0, w, h) for w, h in sizes], seed=105, jitter_deg=10)
    db = DeviceBatch(batch, "cuda:0")
    first, T, n = renderer.forward(db)
    ws, b, s = renderer.ws, db.struct(), stream_ptr()
    for _ in range(2):
        api.rgba_bin_sort(renderer.ctx, b, ws.data_ptr(), ws.numel(), s)
    compare_decisions(batch, oracle.forward(batch, do_render=False), read_intermediates(renderer, db), db)
    img, T2, n2 = torch.empty_like(first), torch.empty_like(T), torch.empty_like(n)
    api.rgba_render_fwd(renderer.ctx, b, ws.data_ptr(), ws.numel(), img.data_ptr(), T2.data_ptr(), n2.data_ptr(), s)
    assert torch.equal(img, first) and torch.equal(T2, T) and torch.equal(n2, n)
