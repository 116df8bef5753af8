"""The profiled figures that bench.py quotes: only those of the lattice it runs, and only
while they were taken on the current kernel sources."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_traffic_is_of_the_size_and_the_sources(tmp_path, monkeypatch):
    f = tmp_path / "t.json"
    d = {"kernel_sources_sha16": bench.kernel_source_hash(),
         "captures": [{"L": 32768, "dram_bytes_per_attempt": 0.34}, {"L": 524288, "dram_bytes_per_attempt": 0.58}]}
    f.write_text(json.dumps(d))
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(f))
    assert bench.profiled_kernel(bench.L)["dram_bytes_per_attempt"] == 0.58
    assert bench.profiled_kernel(32768)["dram_bytes_per_attempt"] == 0.34
    assert bench.profiled_kernel(65536) is None
    f.write_text(json.dumps(dict(d, kernel_sources_sha16="0" * 16)))
    assert bench.profiled_kernel(bench.L) is None
    monkeypatch.setattr(bench, "TRAFFIC_FILE", str(tmp_path / "none.json"))
    assert bench.profiled_kernel(bench.L) is None


def test_committed_captures_are_complete():
    with open(bench.TRAFFIC_FILE) as f:
        d = json.load(f)
    sizes = [c["L"] for c in d["captures"]]
    assert bench.L in sizes and 32768 in sizes
    for c in d["captures"]:
        attempts = c["L"] * c["rows_per_launch"] * c["sweeps_per_launch"]
        assert c["attempts_per_launch"] == attempts
        moved = c["dram_bytes_read_per_launch"] + c["dram_bytes_written_per_launch"]
        assert abs(c["dram_bytes_per_attempt"] * attempts - moved) < 1e-3 * moved
