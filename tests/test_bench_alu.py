"""bench.py's FP64 fraction comes from operations counted on the sources that ran,
or is not given at all."""
import importlib.util
import json
import os

import pytest

from paper_1505_02037_gb300 import traffic_table as TT

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def bench(tmp_path, monkeypatch):
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(mod, "ROOT", str(tmp_path))
    return mod


@pytest.mark.parametrize("stored,want", [("current", True), ("stale", False), ("absent", False)])
def test_fraction_needs_a_current_count(bench, tmp_path, stored, want):
    h = TT.source_hash(TT.COLLIDE_SOURCES) if stored == "current" else "0" * 16
    table = {} if stored == "absent" else {
        "k": {"source_hash": h, "fp64_flops_per_cell": 2000.0, "dram_bytes_per_cell": 1.0}}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(table))
    got = bench.fp64_alu("k", 10 ** 6, 4.0, 1.0)
    if want:
        assert got["achieved_tflops"] == pytest.approx(0.5) and got["frac"] == pytest.approx(0.5)
        assert got["flops_per_cell"] == 2000.0
    else:
        assert got is None
