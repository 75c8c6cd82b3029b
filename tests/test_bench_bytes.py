"""The bench's byte models of the wave steps: the medium is charged once for
all shots."""
import pytest

import bench


def test_shots_share_the_medium():
    # own fields per shot-point, medium per point
    assert bench.step_bytes("rtm", 1) == 16 and bench.step_bytes("rtm", 8) == 12.5
    assert bench.step_bytes("grad", 1) == 72 and bench.step_bytes("grad", 2) == 58
    assert bench.step_bytes("vti", 4) == 26
    assert bench.step_bytes("tti", 2) == 66
    # what perf's cases call the least a forward or VTI step moves, per point
    for s in (1, 2, 8):
        assert bench.step_bytes("rtm", s) * s == 12 * s + 4
        assert bench.step_bytes("vti", s) * s == 24 * s + 8


def test_no_fraction_above_the_measured_peak():
    # 8 x 512^3 at 425 G point-steps/s, which 16 B per shot-point put at 100 %
    assert 425e9 * bench.step_bytes("rtm", 8) / 6798.9e9 == pytest.approx(0.781, abs=1e-3)
