"""The autotuner's table on a stand-in device: one timing per distinct choice of kernels, shared by the staging sizes
that select the same ones, so that their order in the table is no accident of the clock."""
import types

import pytest

from paper_2503_12886_gb300 import batching, synth


class FakeEvent:
    clock = 0.0

    def __init__(self, enable_timing=False):
        self.t = None

    def record(self):
        self.t = FakeEvent.clock

    def elapsed_time(self, other):
        return other.t - self.t


@pytest.mark.parametrize("sizes,runs", [((64, 128, 256), 4), ((256, 128), 2), ((64, 0), 2)])
def test_same_kernels_are_timed_once(monkeypatch, sizes, runs):
    made, ms = [], iter([5.0, 3.0, 7.0, 4.0])

    class FakeBatch:
        def __init__(self, batch, device, tile, smem_batch, models):
            made.append((tile, smem_batch))
            self.models, self.total_pix, self.ms = models, 4, next(ms)

        def pack_images(self, imgs):
            return types.SimpleNamespace(device="cpu")

    def step(db, tg, kind, img):
        FakeEvent.clock += db.ms

    monkeypatch.setattr(batching, "DeviceBatch", FakeBatch)
    monkeypatch.setattr(batching.torch.cuda, "Event", FakeEvent)
    monkeypatch.setattr(batching.torch.cuda, "synchronize", lambda *a: None)
    batch = synth.make_batch([synth.make_model(211, 8, 1)], [synth.Frame(0, 16, 16)], seed=211)
    res = batching.autotune(types.SimpleNamespace(device=0, step=step), batch, [], steps=2, smem_batches=sizes)
    assert len(made) == runs and len(res.table) == 2 * len(sizes)
    assert res.ms == pytest.approx(min(res.table.values()))
    if len(sizes) == 3:  # 64: 5 and 7 ms; 128 and 256: 3 and 4 ms
        assert res.table == pytest.approx({"16x16/64": 5, "16x16/128": 3, "16x16/256": 3, "8x32/64": 7, "8x32/128": 4,
                                           "8x32/256": 4})
        assert (res.tile, res.smem_batch) == ((16, 16), 128)
