"""bench.py quotes a kernel's profiled DRAM traffic only while every file that the traffic follows from is as it
was at the capture (no GPU needed)."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2609_23733_gb300", "csrc")


@pytest.mark.parametrize("kernel", ["attn_full", "gemm"])
def test_traffic_is_dropped_when_a_source_changes(kernel, tmp_path, monkeypatch):
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / f"{kernel}_traffic.txt").write_text(
        f"# a capture\nsource_sha256_16={bench.source_hash(kernel)}\ndram_bytes_per_launch_scaled=1234\n")
    assert bench.traffic_from_profile(kernel) == 1234.0
    sources = {"attn_full": ["attn_full.cu", "attn_plan.cuh", "attn_split.h"], "gemm": ["gemm.cu"]}[kernel]
    for name in sources:
        path = tmp_path / CSRC / name
        text = path.read_text()
        path.write_text(text + "\n// changed\n")
        assert bench.traffic_from_profile(kernel) is None, name
        path.write_text(text)
    assert bench.traffic_from_profile(kernel) == 1234.0
