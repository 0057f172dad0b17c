"""Tile lists at the edges of the sort's paths (shared memory up to 8,192 keys, by positions up to
12,288, through global memory beyond), with and without a depth bucket too crowded for the rank
placement: every list bit for bit against the oracle's."""
import dataclasses
import math

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


def one_tile(n, crowd):
    """n small Gaussians inside one 16 x 16 tile of a 64 x 64 frame: one list of n keys. crowd: that
    many of them at nearly one depth (steps of about two ulps)."""
    m = synth.make_model(71, n, 1, radii=(0.03, 0.03, 0.1), sd_dmean=0.0, log_scale_mu=math.log(1e-4))
    g0 = m.g0.copy()
    g0[0:2, :n] -= 0.107
    if crowd:
        g0[2, :crowd] = 0.02 + 2.4e-7 * np.arange(crowd)
    return synth.make_batch([dataclasses.replace(m, g0=g0)], [synth.Frame(0, 64, 64)], seed=71)


@pytest.mark.parametrize("n,crowd", [(8192, 0), (8193, 0), (12288, 0), (12289, 0), (12289, 900), (33001, 0),
                                     (33001, 900)])
def test_long_lists_sort_like_the_oracle(renderer, n, crowd):
    batch = one_tile(n, crowd)
    r, db, img, T, nc = run_gpu_forward(batch, (16, 16), 64, renderer)
    inter = read_intermediates(r, db)
    assert int(np.diff(inter["tile_start"].astype(np.int64)).max()) == n
    compare_decisions(batch, oracle.forward(batch, do_render=False), inter, db)
