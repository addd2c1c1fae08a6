"""bench.py reports the DRAM traffic of a committed capture for the sources it was
taken on, and none otherwise."""
import pytest


@pytest.mark.parametrize("captured, reported", [("present", 45.0), ("not-kept", None)])
def test_traffic_belongs_to_the_captured_sources(tmp_path, monkeypatch, captured, reported):
    import bench
    summary = tmp_path / "traffic.txt"
    sha = bench.source_sha() if captured == "present" else captured
    summary.write_text(f"# a capture\nsource_sha {sha}\nworkload crossing_batch\nk_row 45\n")
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(summary))
    assert bench.ncu_traffic("k_row", "crossing_batch") == reported


def test_the_committed_summary_without_its_sources_is_not_reported():
    import bench
    text = open(bench.TRAFFIC_FILE).read()
    if "not figures of the present kernels" in " ".join(text.replace("#", " ").split()):
        assert all(bench.ncu_traffic(f, "crossing_batch") is None for f in ("k_row", "k_col", "k_rk"))
