"""Frames of more tiles than a binning CTA has counters are binned in windows of tile rows: offsets and lists
bit for bit against the oracle's for frames of one to six windows, with rectangles within a window, across
their edges and over the whole frame, on either side of frames of one window in the same batch."""
import dataclasses

import numpy as np
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


# windows: 1, 2 of which the last is one row, 2, 6, 6 of 24 rows
@pytest.mark.parametrize("tile,size", [((16, 16), (2048, 1536)), ((16, 16), (2048, 1537)), ((16, 16), (1777, 1777)),
                                       ((16, 16), (4096, 4096)), ((8, 32), (4096, 4096))])
@pytest.mark.parametrize("n", [1, 257, 700])
def test_lists_of_several_windows(renderer, n, tile, size):
    m = synth.make_model(161, n, 3)
    g0 = m.g0.copy()
    u = synth.Stream(161, 70).uniform(2 * n).reshape(2, n)
    g0[0:2, :n] = 1.2 * (u - 0.5)  # all over the frame and past its edges
    g0[7:10, : min(n, 3)] = 0.0    # over the whole frame
    g0[7:10, 3:40] = -3.0          # over several rows of tiles
    m = dataclasses.replace(m, g0=g0)
    frames = [synth.Frame(0, 64, 48), synth.Frame(0, *size), synth.Frame(0, 100, 333)]
    batch = synth.make_batch([m], frames, seed=161, jitter_deg=10)
    r, db, _, _, _ = run_gpu_forward(batch, tile, 64, renderer)
    inter = read_intermediates(r, db)
    stats = compare_decisions(batch, oracle.forward(batch, tile=tile, do_render=False), inter, db, tile)
    tiles = -(-size[0] // tile[0]) * -(-size[1] // tile[1])
    assert stats["pairs"] >= tiles
    area = inter["rects"][db.rec_offsets[1]: db.rec_offsets[1] + n].astype(np.int64)
    assert ((area[:, 2] - area[:, 0]) * (area[:, 3] - area[:, 1])).max() == tiles
