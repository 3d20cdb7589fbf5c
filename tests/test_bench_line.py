"""The benchmark's line as printed: what it keeps, and its length."""
import json

import bench


def test_compact_keeps_the_numbers_and_drops_the_rest():
    roof = {"bound": "alu", "kernel": "k", "achieved": 1.23456789, "peak": 1.25, "unit": "TFLOP/s",
            "frac": 0.987654321, "peak_source": "x" * 400, "kernel_ms": 1e3 / 3}
    line = {"metric": bench.METRIC, "value": 13593123.456789, "n_gpus": 1, "roofline": dict(roof),
            "gpu_launches": 123456789, "e2e": {"value": 1e7 / 3, "h2d_bytes_per_step": 2400000},
            "clocks": {"sm_mhz": 2070.0, "reasons": []}, "none": None, "nan": float("nan"),
            "configs": {"a": {"value": 1e6 / 7, "roofline": dict(roof)},
                        "b": {"x": {"fp64_frac": 1 / 3, "roofline": dict(roof)}}}}
    o = bench.compact(line)
    assert o["roofline"]["peak_source"] == roof["peak_source"] and o["roofline"]["achieved"] == 1.23457
    assert o["value"] == 13593100.0 and o["gpu_launches"] == 123456789 and o["none"] is None
    assert o["e2e"] == {"value": 3333330.0, "h2d_bytes_per_step": 2400000} and o["clocks"] == line["clocks"]
    assert o["configs"]["a"] == {"value": 142860.0, "roofline": {
        "bound": "alu", "achieved": 1.2346, "frac": 0.98765, "kernel_ms": 333.33}}
    assert o["configs"]["b"] == {"x": {"fp64_frac": 0.33333}}
    assert line["configs"]["a"]["roofline"] == roof  # (a copy)
    assert len(json.dumps(o)) < len(json.dumps(line)) - 800


def test_the_traffic_record_follows_every_source_of_the_kernel(tmp_path, monkeypatch):
    """An edit of any of the traversal's sources retires the record; other files do not matter."""
    csrc = tmp_path / "paper_1606_03135_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    for f in bench.TRAVERSAL_SOURCES + ("assemble.cu",):
        (csrc / f).write_text("int %s;\n" % f.split(".")[0])
    rec = {"workload": "w", "traversal_code_sha256_16": bench.kernel_source_hash(
        *(str(csrc / f) for f in bench.TRAVERSAL_SOURCES))}
    (tmp_path / "profiles" / "traversal_traffic.json").write_text(json.dumps(rec))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench._traffic_entry("w") == rec and bench._traffic_entry("v") is None
    (csrc / "assemble.cu").write_text("int other;\n")
    assert bench._traffic_entry("w") == rec
    for f in bench.TRAVERSAL_SOURCES:
        text = (csrc / f).read_text()
        (csrc / f).write_text(text + "int more;\n")
        assert bench._traffic_entry("w") is None
        (csrc / f).write_text(text + "// a comment\n")
        assert bench._traffic_entry("w") == rec
