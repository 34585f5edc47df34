"""The recorded DRAM traffic of the force kernel counts only while the sources it was taken from are unchanged."""
import os
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_recorded_traffic_lapses_with_any_of_its_sources(tmp_path, monkeypatch):
    sys.path.insert(0, ROOT)
    import bench
    names = [os.path.basename(f) for f in bench.FORCE_SOURCES]
    assert {"force_launch.cuh", "tile.cuh", "kernels_force.cu"} <= set(names)
    copies = [shutil.copy(f, tmp_path) for f in bench.FORCE_SOURCES]
    rec = tmp_path / "rec.md"
    rec.write_text("- kernel: `k`\n- source_sha: `%s`\n- dram_bytes_per_particle: `143.5`\n" % bench.source_sha(copies))
    monkeypatch.setattr(bench, "FORCE_SOURCES", copies)
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(rec))
    assert bench.recorded_traffic("k", 1000) == 143500
    assert bench.recorded_traffic("other", 1000) is None
    for f in copies:
        text = open(f).read()
        open(f, "a").write("\n")
        assert bench.recorded_traffic("k", 1000) is None
        open(f, "w").write(text)
    assert bench.recorded_traffic("k", 1000) == 143500
