"""The counters that the benchmark takes from a committed profile count as current only while the kernel's
source and every header of it are those they were taken with."""
import os
import shutil

import pytest

import bench

SRC = "paper_1411_6206_gb300/csrc/k_dc_rows.cuh"


@pytest.fixture()
def tree(tmp_path, monkeypatch):
    for d in ("paper_1411_6206_gb300/csrc", "include"):
        shutil.copytree(os.path.join(bench.ROOT, d), tmp_path / d)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles" / "p.txt").write_text(
        f"kernel_source: {SRC}\nsource_sha256: {bench.source_digest(SRC)}\ndram_bytes_per_launch: 123\n")
    return tmp_path


def test_unchanged_sources_keep_the_counters(tree):
    assert bench.profiled_traffic("p.txt") == 123


@pytest.mark.parametrize("name", ["k_dc_rows.cuh", "dc_row_body.cuh", "dft_reg.cuh", "lps_internal.cuh"])
def test_a_changed_source_or_header_drops_them(tree, name):
    p = tree / "paper_1411_6206_gb300" / "csrc" / name
    p.write_text(p.read_text() + "\n// changed\n")
    assert bench.profiled_traffic("p.txt") is None


def test_other_sources_do_not(tree):
    p = tree / "paper_1411_6206_gb300" / "csrc" / "k_lrs.cu"
    p.write_text(p.read_text() + "\n// changed\n")
    assert bench.profiled_traffic("p.txt") == 123
