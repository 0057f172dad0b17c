"""Tile lists at the edges of the sort's instances (up to 2,048, 4,096 and 8,192 keys in shared memory,
a radix sort there up to 4,544, longer lists through global memory), with and without a depth bucket too
crowded for the rank placement: every list bit for bit against the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2503_12886_gb300.rasterizer import Renderer

from gpu_helpers import compare_decisions, read_intermediates, run_gpu_forward
from test_gpu_long_lists import one_tile

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("n,crowd", [(1, 0), (2, 0), (511, 0), (512, 0), (513, 0), (2047, 0), (2048, 0), (2048, 700),
                                     (2049, 0), (4096, 0), (4096, 900), (4097, 0), (4544, 900), (4545, 900), (8191, 0),
                                     (8192, 900), (8193, 900)])
def test_list_lengths_sort_like_the_oracle(renderer, n, crowd):
    batch = one_tile(n, crowd)
    r, db, img, T, nc = run_gpu_forward(batch, (16, 16), 64, renderer)
    inter = read_intermediates(r, db)
    assert int(np.diff(inter["tile_start"].astype(np.int64)).max()) == n
    compare_decisions(batch, oracle.forward(batch, do_render=False), inter, db)
