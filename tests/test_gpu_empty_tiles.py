"""Empty tiles of the forward: four pixels at a time where rows and arrays allow it, else one by one.
The same batch into arrays at 16-byte and at 4-byte boundaries gives the same bits, and the pixels no
Gaussian reaches hold the background, T = 1 and no contributors exactly."""
import pytest
import torch

from paper_2503_12886_gb300 import api, synth
from paper_2503_12886_gb300.rasterizer import DeviceBatch, Renderer, stream_ptr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    import __graft_entry__
    __graft_entry__.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("tile", [(16, 16), (8, 32)])
@pytest.mark.parametrize("sizes", [[(256, 200)], [(61, 33), (64, 64), (66, 50), (130, 97), (128, 36)], [(1, 1), (1000, 3)]])
@pytest.mark.parametrize("n", [1, 400])
def test_background_at_any_alignment(renderer, tile, sizes, n):
    m = synth.make_model(91, n, 3)
    batch = synth.make_batch([m], [synth.Frame(0, w, h) for w, h in sizes], seed=91, jitter_deg=5, random_bg=True)
    db = DeviceBatch(batch, "cuda:0", tile=tile)
    P = db.total_pix
    renderer.forward(db)  # sizes the workspace
    b, s, ws = db.struct(), stream_ptr(), renderer.ws
    target = torch.rand(3 * P + 1, device="cuda:0")
    got = []
    for off in (0, 1):
        img, T, nc = (torch.full((k * P + 1,), -7.0, device="cuda:0") for k in (3, 1, 1))
        nc = nc.to(torch.int32)
        api.rgba_preprocess(renderer.ctx, b, ws.data_ptr(), ws.numel(), s)
        api.rgba_bin_sort(renderer.ctx, b, ws.data_ptr(), ws.numel(), s)
        api.rgba_render_fwd(renderer.ctx, b, ws.data_ptr(), ws.numel(), img[off:].data_ptr(), T[off:].data_ptr(),
                            nc[off:].data_ptr(), s)
        tg, step_img = target[:3 * P].clone(), torch.empty(3 * P + 1, device="cuda:0")
        if off:
            tg = torch.cat([tg[:1], tg])
        rc, out = api.rgba_step(renderer.ctx, b, ws.data_ptr(), ws.numel(), tg[off:].data_ptr(), api.RGBA_LOSS_L1,
                                step_img[off:].data_ptr(), s)
        assert rc == api.RGBA_OK
        lay = renderer.layout(db)
        dl = ws[lay.pix_dl: lay.pix_dl + 12 * P].view(torch.float32).clone()
        got.append((img[off:off + 3 * P], T[off:off + P], nc[off:off + P], step_img[off:off + 3 * P], dl, out.loss))
    for a, c in zip(got[0][:5], got[1][:5]):
        assert torch.equal(a, c)
    assert abs(got[0][5] - got[1][5]) <= 1e-5 * got[0][5]  # per-warp fp32 loss sums, in any order
    img, T, nc, step_img, dl, _ = got[0]
    assert torch.equal(img, step_img)
    for f, (im, t, k) in enumerate(zip(db.image_views(img), db.pix_views(T), db.pix_views(nc))):
        free = k == 0
        assert bool((t[free] == 1).all()) and bool((k >= 0).all())
        bg = db.fparams[f, 17:20]
        assert all(torch.equal(im[c][free], bg[c].expand(int(free.sum()))) for c in range(3))
    scale = [1.0 / (3.0 * w * h * len(sizes)) for w, h in sizes]
    for f, (d, im, tg) in enumerate(zip(db.image_views(dl), db.image_views(img), db.image_views(target[:3 * P]))):
        assert bool((torch.sign(d) == torch.sign(im - tg)).all())
        assert float(d.abs().max()) == pytest.approx(scale[f], rel=1e-6)
