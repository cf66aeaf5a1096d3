"""bench.py takes DRAM traffic from a committed profile only while every source
of the profiled kernel is the one it was captured from."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.fixture
def tree(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2303_11811_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (tmp_path / "profiles").mkdir()
    for f in ("lbm_kernels.cu", "fixed64.cuh", "df.cuh"):
        (csrc / f).write_text("// " + f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / "k.md").write_text(
        f"source_sha256_16: {bench.source_hash(*bench.kernel_sources())}\n"
        "dram_bytes_per_cell: 400\n")
    return csrc


def test_unchanged(tree):
    assert bench.profiled_traffic("k", 1000) == 400 * 1000
    assert bench.profiled_traffic("other", 1000) is None


@pytest.mark.parametrize("f", ["lbm_kernels.cu", "fixed64.cuh", "df.cuh"])
def test_changed_source(tree, f):
    (tree / f).write_text("// another")
    assert bench.profiled_traffic("k", 1000) is None
