"""The recorded DRAM traffic of the tile kernel is used only while every source it
depends on is the one it was recorded with."""
import json
import os

import pytest

import bench

CSRC = os.path.join("paper_1407_1810_gb300", "csrc")


def _tree(tmp_path, monkeypatch):
    root = bench.ROOT
    (tmp_path / CSRC).mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    for f in ("tiles_one.cu", "tiles_two.cu", "tiles32.cuh", "particles32.cu"):
        (tmp_path / CSRC / f).write_bytes(open(os.path.join(root, CSRC, f), "rb").read())
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / "k_tiles32_traffic.json").write_text(
        json.dumps({"dram_bytes_per_particle": 52.5, "source_sha256_16": bench.traffic_hash()}))


@pytest.mark.parametrize("changed", ["tiles_two.cu", "tiles32.cuh", "particles32.cu"])
def test_a_changed_source_retires_the_record(tmp_path, monkeypatch, changed):
    _tree(tmp_path, monkeypatch)
    assert bench.recorded_traffic() == 52.5
    with open(tmp_path / CSRC / changed, "a") as f:
        f.write("// changed\n")
    assert bench.recorded_traffic() is None


def test_no_record(tmp_path, monkeypatch):
    _tree(tmp_path, monkeypatch)
    os.remove(tmp_path / "profiles" / "k_tiles32_traffic.json")
    assert bench.recorded_traffic() is None
