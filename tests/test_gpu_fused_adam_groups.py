"""The fused Adam update at the edges of its frame groups (eight or sixteen frames of a model), against the separate
calls: one step from zero moments, compared as in test_gpu_fused_adam.py, whose reasons and tolerances hold here:
the compositing backward's atomics make the gradients differ in their last bits, so parameters and
moments are compared where |g| is above 1e-4 of the tensor's largest. Blendshape counts past the 32 that one pass of the
products covers, and Gaussian counts that do not fill the last 32."""
import pytest
import torch

from paper_2503_12886_gb300 import api, synth
from paper_2503_12886_gb300.optim import Adam
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer

import test_gpu_fused_adam as base

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("bound", [False, True])
@pytest.mark.parametrize("nb,k,n", [(8, 8, 3001), (9, 33, 2052), (16, 16, 3003), (16, 40, 1000)])
def test_fused_update_at_group_edges(renderer, nb, k, n, bound):
    mesh = synth.make_head_mesh(8, 12, 24) if bound else None
    models = [synth.make_bound_model(201, n, k, mesh) if bound else synth.make_model(201, n, k),
              synth.make_model(202, 500, 5, mask=synth.MASK_PAPER)]
    frames = [synth.Frame(0, 64, 80, synth.frame_verts(mesh, 201, f) if bound else None) for f in range(nb)]
    batch = synth.make_batch(models, frames + [synth.Frame(1, 48, 64)] * 3, seed=201, jitter_deg=15, random_bg=True)
    targets = synth.make_targets(batch, 3)
    dbA, dbB = DeviceBatch(batch, "cuda:0"), DeviceBatch(batch, "cuda:0", grads=False)
    dbB.grad_psi = torch.zeros_like(dbB.psi)
    optA, optB = Adam(renderer, dbA), Adam(renderer, dbB)
    wsA, wsB = base._workspace(dbA), base._workspace(dbB)
    imgA = torch.empty(3 * dbA.total_pix, device="cuda:0")
    imgB = torch.empty_like(imgA)
    p0 = [(m.g0.clone(), m.dg.clone()) for m in dbA.models]
    base._separate(renderer, dbA, optA, wsA, dbA.pack_images(targets), imgA)
    optB.train_step(wsB, dbB.pack_images(targets), api.RGBA_LOSS_L1, imgB)
    torch.cuda.synchronize()
    (ovA, lossA), (ovB, lossB) = base._counters(dbA, wsA), base._counters(dbB, wsB)
    assert ovA == 0 and ovB == 0 and abs(lossA - lossB) <= 1e-5 * abs(lossA)
    assert torch.equal(imgA, imgB)
    torch.testing.assert_close(dbB.grad_psi, dbA.grad_psi, rtol=1e-3, atol=1e-7)
    for mi, (mA, mB) in enumerate(zip(dbA.models, dbB.models)):
        for pA, pB, p, g, momA, momB in ((mA.g0, mB.g0, p0[mi][0], mA.grad_g0, optA.m[mi][0], optB.m[mi][0]),
                                         (mA.dg, mB.dg, p0[mi][1], mA.grad_dg, optA.m[mi][1], optB.m[mi][1])):
            sig = g.abs() > 1e-4 * g.abs().max()
            assert int(sig.sum()) > 0
            torch.testing.assert_close(pB[sig], pA[sig], rtol=0, atol=1e-6)
            assert bool((pB[sig] != p[sig]).any()) and torch.equal(pB[g == 0], pA[g == 0])
            torch.testing.assert_close(momB[sig], momA[sig], rtol=1e-3, atol=1e-6 * float(g.abs().max()))
    assert int(optA.step_dev.item()) == int(optB.step_dev.item()) == 1
