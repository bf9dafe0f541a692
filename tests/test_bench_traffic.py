"""The traffic record that bench.py reports parses, holds what it reads, and carries the whole command that made it."""
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_modal_tail_traffic_record():
    d = json.load(open(os.path.join(ROOT, "profiles", "modal_tail_traffic_128cube.txt")))
    assert d["launches"] == [r + w for r, w in zip(d["dram_bytes_read"], d["dram_bytes_written"])]
    assert d["dram_bytes_per_launch"] == sum(d["launches"]) / len(d["launches"])
    assert len(d["source_hash"]) == 16 and d["sources"] == ["modal.cuh", "modal_inst.cu"]
    assert "python -m paper_1212_6680_gb300.profile_case fpcg" in d["command"]
