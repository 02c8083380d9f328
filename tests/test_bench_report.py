"""bench.py reports the pair kernels that ran, whatever their rate."""
import pytest

import bench

PEAK = 4.0e13


def _tm(pairs, ms, launches=2):
    return dict(pair_energy_ms=ms * launches, pair_energy_launches=launches,
                pair_energy_pairs=pairs * launches, pair_force_ms=ms * launches,
                pair_force_launches=launches, pair_force_pairs=pairs * launches)


# 4.3e9 pairs in 2.345 ms: 3.3e13 operations a second at 18 per pair, below
# the peak; and a rate far above it
@pytest.mark.parametrize("pairs,ms", [(4.3e9, 2.345), (1.1e12, 60.0)])
def test_hierarchical_sums_are_named(pairs, ms):
    tm = _tm(pairs, ms)
    f = bench.fields_roofline(tm, "hierarchical", PEAK, "", None)
    g = bench.force_roofline(tm, "hierarchical", PEAK, None)
    assert f["kernel"].startswith("tree_") and g["kernel"].startswith("tree_")
    for r in (f, g):
        assert r["frac"] is None and r["achieved"] is None
        assert r["covered_pairs_per_s"] == pytest.approx(pairs / (ms * 1e-3))


def test_direct_sums_are_named():
    tm = _tm(4.3e9, 4.0)
    f = bench.fields_roofline(tm, "direct", PEAK, "basis", None)
    g = bench.force_roofline(tm, "direct", PEAK, None)
    assert f["kernel"] == "pair_energy_grid" and g["kernel"] == "pair_force_grid"
    rate = 4.3e9 / 4.0e-3
    assert f["frac"] == pytest.approx(rate * bench.OPS_PER_PAIR / PEAK)
    assert g["frac"] == pytest.approx(rate * bench.FORCE_OPS_PER_PAIR / PEAK)
    assert bench.force_roofline(dict(tm, pair_force_launches=0), "direct", PEAK, None) is None
