"""A captured DRAM traffic is reported only for the labelling tile it was
captured with, where its line names one."""
import bench


def test_traffic_of_the_tile_in_use(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: "cafe")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / "traffic.txt").write_text("k 2.0 cafe 8x8x4\nk 3.0 cafe 8x4x8\nk 9.0 beef 8x8x8\nj 5.0 cafe\n")
    assert bench.committed_traffic("k", 10, [8, 8, 4]) == 20.0
    assert bench.committed_traffic("k", 10, (8, 4, 8)) == 30.0
    assert bench.committed_traffic("k", 10, (8, 8, 8)) is None
    assert bench.committed_traffic("j", 10, (8, 8, 8)) == 50.0
    assert bench.committed_traffic("k", 10) == 20.0
