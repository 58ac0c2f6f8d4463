"""The committed FP64 instruction counts are used only while every source that
holds counted arithmetic is the one they were taken on."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("name", ["bulk.cu", "collide.cuh", "fix64.cuh", "lbm_internal.cuh"])
def test_counts_lapse_when_a_counted_source_changes(name, tmp_path, monkeypatch):
    csrc = os.path.join("paper_2307_16766_gb300", "csrc")
    shutil.copytree(os.path.join(ROOT, csrc), tmp_path / csrc)
    shutil.copytree(os.path.join(ROOT, "profiles"), tmp_path / "profiles")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.bulk_fp64_flops() is not None
    with open(tmp_path / csrc / name, "a") as f:
        f.write("// changed\n")
    assert bench.bulk_fp64_flops() is None
