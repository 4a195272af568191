"""bench.py's shares of the HBM peak count the bytes that the launches of a call move."""
import pytest

import bench


def launches(storage, **n):
    return {k: {"launches": v, "algorithmic_bytes_per_node": bench.BYTES[storage][1][k]} for k, v in n.items()} | {
        "boundary_kernel": {"launches": 1}}


@pytest.mark.parametrize("storage,n,moved", [
    (0, dict(moment_kernel=1, advance_kernel=99, collide_kernel=1), (99 * 112 + 2 * 272) / 100),
    (0, dict(moment_kernel=100, collide_kernel=100), 544),
    (0, dict(step_kernel=100), 448),
    (2, dict(moment_kernel=100, collide_kernel=100), 192 + 176),
])
def test_shares_of_the_peak(storage, n, moved):
    peak = (6703.8, "measured")
    s = bench.hbm_shares(5000.0, launches(storage, **n), storage, 100, peak)
    assert s["bytes_per_node_design"] == pytest.approx(moved)
    assert s["hbm_pct_of_peak"] == pytest.approx(100 * 5000e6 * moved / 6703.8e9)
    assert s["hbm_pct_of_peak_populations"] == pytest.approx(100 * 5000e6 * bench.BYTES[storage][0] / 6703.8e9)


def test_the_multi_step_path_stays_below_the_peak():
    """At its measured rate the step that keeps its populations on the chip takes a third of the peak."""
    s = bench.hbm_shares(22785.0, launches(0, moment_kernel=1, advance_kernel=99, collide_kernel=1), 0, 100, (6703.8, "measured"))
    assert 30 < s["hbm_pct_of_peak"] < 50 and s["hbm_pct_of_peak_populations"] > 100
