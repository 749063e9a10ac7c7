"""bench.py's DRAM bytes per launch: from captures of the kinds of launch that the profiled entry holds,
and none where a kind was not captured or the kernel source has changed since (CPU only)."""
import json

import pytest

import bench


@pytest.fixture
def captures(tmp_path, monkeypatch):
    d = {"source_sha256": "x", "f32": {"dram_bytes": 110, "algorithmic_bytes": 100},
         "f32_norm": {"dram_bytes": 120, "algorithmic_bytes": 100},
         "f32_resid": {"dram_bytes": 130, "algorithmic_bytes": 150}, "f16": {"dram_bytes": 98, "algorithmic_bytes": 100}}
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "dslash32_traffic.json").write_text(json.dumps(d))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: "x")


def test_kinds_of_a_step(captures, monkeypatch):
    assert bench.step_kinds("f32", "f16") == ["f32_norm", "f32_resid"]
    assert bench.measured_traffic(bench.step_kinds("f32", "f16"), 1000.0) == 1000.0     # 250 / 250
    assert bench.measured_traffic(["f32"], 1000.0) == pytest.approx(1100.0)
    assert bench.measured_traffic(bench.step_kinds("f16", "f16"), 1000.0) is None       # no capture of f16_cheb
    assert bench.measured_traffic(bench.step_kinds("f32", "f32"), 1000.0) is None       # a mixture
    assert bench.measured_traffic(bench.step_kinds("f64", "f16"), 1000.0) is None
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: "y")
    assert bench.measured_traffic(["f32"], 1000.0) is None
