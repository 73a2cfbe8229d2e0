"""Host test: a profiled DRAM figure lapses with any source its profile names."""
import hashlib

import bench


def test_traffic_needs_every_named_source(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    lines = ["dram_bytes_per_iteration: 5"]
    for name in ("k.cu", "k.cuh"):
        (tmp_path / name).write_text(name)
        lines.append(f"source_sha1 ({name}): {hashlib.sha1(name.encode()).hexdigest()}")
    (tmp_path / "profiles" / "p.md").write_text("\n".join(lines))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    figure = lambda: bench._profiled_traffic("p.md", "k.cu", "dram_bytes_per_iteration")
    assert figure() == 5.0
    assert bench._profiled_traffic("p.md", "other.cu", "dram_bytes_per_iteration") is None
    (tmp_path / "k.cuh").write_text("changed")
    assert figure() is None
    (tmp_path / "k.cuh").unlink()
    assert figure() is None
