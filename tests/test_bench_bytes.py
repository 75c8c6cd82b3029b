"""The bench's byte models of the wave steps: the medium is charged once for
all shots, and a captured traffic figure is used only for as many shots as it
was taken with and while the launch planner that decides the halo re-reads is
the one captured."""
import json
import os

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


def test_traffic_belongs_to_its_number_of_shots(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    csrc = tmp_path / "paper_2507_11067_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (csrc / "k.cu").write_text("__global__ void k() {}\n")
    h = {"k.cu": bench.code_hash(str(csrc / "k.cu"))}
    recs = {"wave": {"dram_bytes_per_point": 13.0, "shots": 8, "sources": h},
            "sweep": {"dram_bytes_per_point": 8.0, "sources": h}}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(recs))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.captured_traffic("wave", 10, 8) == 130.0
    assert bench.captured_traffic("wave", 10, 2) is None
    assert bench.captured_traffic("wave", 10) is None
    assert bench.captured_traffic("sweep", 10) == 80.0


def test_captures_cover_the_launch_planner():
    t = json.load(open(os.path.join(bench.ROOT, "profiles", "traffic.json")))
    for key, rec in t.items():
        if not key.startswith("f64"):       # (the FP64 sweeps' grids are their own)
            assert "abi.cu" in rec["sources"], key
        assert key.split()[0] in ("wave_fwd", "wave_adj_scaled", "vti_fwd", "tti_fwd") or "shots" not in rec, key
        if "fwd" in key or "adj" in key:
            assert rec["shots"] >= 1, key
