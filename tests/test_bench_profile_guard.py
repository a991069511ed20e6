"""The bench quotes captured counters only while every source of the kernel is
the one they were taken on (CPU)."""
import json
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_1909_01589_gb300", "csrc")


@pytest.fixture
def tree(tmp_path, monkeypatch):
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return tmp_path


def _included(csrc, name, seen):
    seen.add(name)
    for line in open(csrc / name):
        if line.startswith("#include \""):
            other = line.split('"')[1]
            if other not in seen and (csrc / other).exists():
                _included(csrc, other, seen)
    return seen


def test_every_source_counts(tree):
    record = tree / "profiles" / "k_interval_df64_ne4096_traffic.json"
    record.write_text(json.dumps({"dram_bytes_per_launch": 1.0, "kernel_sha256": bench._kernel_hash()}))
    assert bench._read_profile("df64")["dram_bytes_per_launch"] == 1.0
    assert bench._read_profile("fp32") is None
    for name in sorted(_included(tree / CSRC, "lrdmc_kernels.cu", set())):
        path = tree / CSRC / name
        text = path.read_text()
        path.write_text(text + "\n")
        assert bench._read_profile("df64") is None, name
        path.write_text(text)
    assert bench._read_profile("df64") is not None
