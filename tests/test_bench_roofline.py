"""What bench.py calls a fraction of a peak is one: counted from what the kernel
executes, none where there is no capture of the present kernel, and never above
1 in the committed captures and bench lines."""
import glob
import json
import os

import pytest

import bench
from conftest import ROOT

PEAK = 152 * bench.ISSUE_PER_SM * 2070 / 1e3  # the captures' device at its highest clock


def _line(capture, units, ms, sources=bench.SCAN_SOURCES):
    return bench.roofline_obj("k", "unit", units, ms, 2, 2 * ms, PEAK, 152, 2070, "test", capture, sources)


@pytest.mark.parametrize("name,sources", [
    ("k_scan_lanes_traffic.json", bench.SCAN_SOURCES), ("k_scan_lanes_l201_traffic.json", bench.SCAN_SOURCES),
    ("k_scan_lanes_mesh_traffic.json", bench.SCAN_SOURCES), ("k_grid_lines_traffic.json", bench.GRID_SOURCES)])
def test_captured_launch_is_a_fraction(name, sources):
    t = json.load(open(os.path.join(ROOT, "profiles", name)))
    assert t["source_sha"] == bench.scan_source_hash(sources)  # of the present kernel
    r = _line(name, t["valid_samples"], t["duration_us"] / 1e3, sources)
    assert r["achieved"] == pytest.approx(t["warp_instructions"] / t["duration_us"] / 1e3)
    assert 0.3 < r["frac"] <= 1.0
    assert r["traffic"] == pytest.approx(t["dram_bytes"] / 2)
    half = _line(name, t["valid_samples"] / 2, t["duration_us"] / 1e3, sources)
    assert half["frac"] == pytest.approx(r["frac"] / 2)


def test_no_fraction_without_a_capture(monkeypatch):
    for r in (_line(None, 1e9, 1.0), _line("missing.json", 1e9, 1.0)):
        assert r["achieved"] is None and r["frac"] is None and r["traffic"] is None
        assert r["every_unit"]["tflops"] == pytest.approx(30 * 1e9 / 1e-3 / 1e12)
    monkeypatch.setattr(bench, "scan_source_hash", lambda *a: "another kernel")
    assert _line("k_scan_lanes_traffic.json", 1e9, 1.0)["frac"] is None


def _fracs(o, path=""):
    if isinstance(o, dict):
        for k, v in o.items():
            if k.startswith("frac") and isinstance(v, float):
                yield path + "." + k, v
            yield from _fracs(v, path + "." + k)


def test_committed_lines_hold_no_fraction_above_one():
    found = 0
    for f in glob.glob(os.path.join(ROOT, "profiles", "*bench*.json")):
        for ln in open(f):
            if ln.startswith("{") and ln.rstrip().endswith("}"):
                for k, v in _fracs(json.loads(ln)):
                    found += 1
                    assert v <= 1.0, (os.path.basename(f), k, v)
    assert found > 0
