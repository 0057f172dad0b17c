"""The Gaussian backward at the edges of its frame groups (eight or sixteen frames), blendshape
blocks (16 and 32) and chunks (32 Gaussians): gradients against the oracle's, whose dL/dimg is zeroed
at the pixels it flags as ambiguous, within the workload's gradient tolerance."""
import numpy as np
import pytest
import torch

from paper_2503_12886_gb300 import synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer

from gpu_helpers import backward_errors, oracle_fwd_bwd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("bound", [False, True])
@pytest.mark.parametrize("nb,k,n", [(1, 1, 31), (7, 16, 65), (8, 17, 96), (9, 32, 33), (16, 33, 100), (17, 5, 130)])
def test_gradients_at_group_edges(renderer, nb, k, n, bound):
    mesh = synth.make_head_mesh(8, 12, 24) if bound else None
    models = [synth.make_bound_model(81, n, k, mesh) if bound else synth.make_model(81, n, k),
              synth.make_model(82, 40, max(1, k // 2))]
    verts = [synth.frame_verts(mesh, 81, f) if bound else None for f in range(nb)]
    batch = synth.make_batch(models, [synth.Frame(0, 40, 48, v) for v in verts] + [synth.Frame(1, 48, 40)], seed=81,
                             jitter_deg=10, random_bg=True)
    targets = synth.make_targets(batch, 83)
    _, _, dls, per_model, dpsi, _ = oracle_fwd_bwd(batch, targets, "l2", drop_flagged=True)
    db = DeviceBatch(batch, "cuda:0")
    img, T, nc = renderer.forward(db)
    renderer.backward(db, db.pack_images(dls), T, nc)
    torch.cuda.synchronize()
    errs = backward_errors(batch, db, per_model, dpsi)
    assert np.isfinite(list(errs.values())).all() and max(errs.values()) <= 1.0, errs
