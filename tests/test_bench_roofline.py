"""bench.py's compositing rates credit no work that the kernel does not do: entries that the block masks drop count
nowhere, and rejected evaluations only in the figure that says so."""
import pytest

import bench


@pytest.mark.parametrize("comp", ["render_bwd", "render_step"])
def test_dropped_units_are_not_credited(comp):
    stats = {"bwd_pairs": 1000, "bwd_hits": 100, "fwd_hits": 110}
    few, many = (bench.compositing_rates(comp, 1e-6, units, stats) for units in (2000, 2_000_000))
    assert few["blended"] == many["blended"] and few["evaluated"] == many["evaluated"]
    assert many["blended"] < many["evaluated"] < many["table"]
    per_unit = bench.BWD_FLOPS_PER_UNIT + (bench.FWD_FLOPS_PER_UNIT if comp == "render_step" else 0)
    rejected = 32 * 100 - 1000 if comp == "render_bwd" else 32 * 210 - 2000
    assert many["blended"] == pytest.approx(1000 * per_unit * 1e-6)
    assert many["evaluated"] == pytest.approx((1000 * per_unit + 9 * rejected) * 1e-6)


def test_blending_everywhere_rejects_nothing():
    rate = bench.compositing_rates("render_bwd", 1.0, 3200, {"bwd_pairs": 3200, "bwd_hits": 100, "fwd_hits": 0})
    assert rate["blended"] == rate["evaluated"] == rate["table"]
