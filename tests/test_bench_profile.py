"""The bench takes the figures of an ncu summary only while every file that the solve kernel
is made of is as it was then."""
import os
import shutil

import pytest

import bench

FILES = ("mh_kernels.cu", "mh_levels.cuh", "mh_barrier.h", "mh_internal.h")


@pytest.fixture
def tree(tmp_path, monkeypatch):
    csrc = tmp_path / "paper_2603_16721_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for name in FILES:
        shutil.copy(os.path.join(bench.ROOT, "paper_2603_16721_gb300", "csrc", name), csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "k_solve_c2.md").write_text(
        f"# k_solve\n\n- `kernel_source_sha256: {bench.kernel_source_sha256()}`\n- `dram_bytes_per_launch: 7`\n")
    return csrc


def test_an_unchanged_source_gives_the_figures(tree):
    assert bench._profiled_fields()["dram_bytes_per_launch"] == "7"


@pytest.mark.parametrize("name", FILES)
def test_a_change_in_any_file_drops_them(tree, name):
    with open(tree / name, "a") as f:
        f.write("\n// changed\n")
    assert bench._profiled_fields() == {}
