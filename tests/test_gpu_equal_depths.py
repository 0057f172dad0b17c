"""Tile lists with groups of exactly equal depths, where only the Gaussian index decides the order: in buckets that the
rank placement takes, and in crowded ones through the radix sorts in shared memory (up to 8,192 keys) and in
global memory, there with runs that the tie pass orders (up to 32) and longer ones. The depths' spread sets the number
of radix passes, odd and even, and with it the buffer the result lies in. Every list bit for bit against the oracle's;
the block masks that travel with the keys give the image of lists without them."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer

from gpu_helpers import compare_decisions, read_intermediates, run_gpu_forward
from test_gpu_block_masks import behind

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


def grouped(n, group, spread):
    """n small Gaussians inside one tile of a 64 x 64 frame, depths within `spread`; the depths of the first 2,700
    repeat in groups, whose members lie 3 (mod n) indices apart."""
    m = synth.make_model(181, n, 1, mask=0x7, radii=(0.03, 0.03, 0.1), sd_dmean=0.0, log_scale_mu=math.log(1e-4))
    g0 = m.g0.copy()
    g0[0:2, :n] -= 0.107
    z = (spread * (synth.Stream(181, 70).uniform(n) - 0.5)).astype(np.float32)
    for s in range(0, min(n, 2700) // group * group, group):
        z[s: s + group] = z[s]
    g0[2, :n] = z[(3 * np.arange(n)) % n if n % 3 else np.arange(n)]
    return synth.make_batch([dataclasses.replace(m, g0=g0)], [synth.Frame(0, 64, 64)], seed=181)


@pytest.mark.parametrize("spread", [0.1, 1.5e-3, 6e-6])
@pytest.mark.parametrize("group", [20, 33, 900])
@pytest.mark.parametrize("n", [2047, 4545, 8192, 8194, 33001])
def test_groups_of_equal_depths(renderer, n, group, spread):
    batch = grouped(n, group, spread)
    r, db, img, T, nc = run_gpu_forward(batch, (16, 16), 64, renderer)
    inter = read_intermediates(r, db)
    assert int(np.diff(inter["tile_start"].astype(np.int64)).max()) == n
    depths = np.unique(inter["records"][:n, 9], return_counts=True)[1]
    assert depths.max() >= group
    compare_decisions(batch, oracle.forward(batch, do_render=False), inter, db)


@pytest.mark.parametrize("n,group,spread", [(4545, 900, 0.1), (8192, 33, 6e-6), (8194, 20, 1.5e-3), (33001, 900, 0.1),
                                            (33001, 33, 6e-6)])
def test_masks_travel_with_the_keys(renderer, n, group, spread):
    batch = grouped(n, group, spread)
    got = [renderer.forward(DeviceBatch(batch, "cuda:0", models=m)) for m in (None, [behind(batch.models[0], "cuda:0")])]
    renderer.ws = None
    assert int((got[0][2] > 0).sum()) > 0
    for a, b in zip(*got):
        assert torch.equal(a, b)
