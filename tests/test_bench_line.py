"""The benchmark's line as printed: what it keeps, and its length."""
import json

import bench


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
