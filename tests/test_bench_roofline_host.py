"""The roofline part of bench.py's line: executed FP32 operations against the FP32 peak, instructions
against the issue rate and DRAM bytes come from counters of the kernel's present sources, and are left out,
with the reason, for other sources or workloads."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.fixture
def counters(monkeypatch, tmp_path):
    with open(bench.VOIGT_COUNTERS) as f:
        d = json.load(f)

    def put(digest):
        path = tmp_path / "counters.json"
        path.write_text(json.dumps(dict(d, sources_sha256=digest)))
        monkeypatch.setattr(bench, "VOIGT_COUNTERS", str(path))
        return d["launches"]
    return put


@pytest.mark.parametrize("kind,ms", [("exomol", 3.3), ("large", 335.0)])
def test_fractions_of_both_peaks(counters, kind, ms):
    c = counters(bench.voigt_sources_digest())[kind]
    evals = c["evaluations"] * (1 if kind == "exomol" else 10)
    r = bench.voigt_roofline(evals, ms, kind, 152, {"sm_mhz": 2070.0}, {"measured_tflops": 78.5})
    assert r["unit"] == "T warp instructions/s" and 0.3 < r["frac"] < 1.0
    f = r["fp32"]
    assert f["peak"] == pytest.approx(80.55, abs=0.01) and f["frac"] == pytest.approx(f["achieved"] / f["peak"])
    assert 0.2 < f["frac"] < f["frac_of_measured"] < 1.0
    assert r["traffic"] == pytest.approx(c["dram_bytes"] * evals / c["evaluations"])


def test_other_sources_and_workloads_are_not_reported(counters):
    counters("0" * 64)
    for kind, why in (("large", "sources changed"), (None, "no counters")):
        r = bench.voigt_roofline(1e13, 300.0, kind, 152, {}, {"measured_tflops": 78.5})
        assert r["achieved"] is None and r["frac"] is None and r["traffic"] is None and r["fp32"]["frac"] is None
        assert why in r["note"] and r["kernel_ms"] == 300.0
