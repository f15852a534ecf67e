"""The hash that ties stored counters to the search kernel covers every file
that fixes the measured kernel: its instances too, and a missing one is another kernel."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_1603_09320_gb300", "csrc")


@pytest.fixture
def tree(tmp_path, monkeypatch):
    os.makedirs(tmp_path / CSRC)
    for f in os.listdir(os.path.join(bench.ROOT, CSRC)):
        if f.startswith("search"):
            shutil.copy(os.path.join(bench.ROOT, CSRC, f), tmp_path / CSRC / f)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return tmp_path / CSRC


@pytest.mark.parametrize("name", ["search.cu", "search_kernel.cuh", "search_dev.cuh", "search_pick.cuh", "search_f32.cu",
                                  "search_bf16.cu", "search_f16.cu", "search_fp8.cu"])
def test_hash_covers_the_kernel_and_its_instances(tree, name):
    before = bench.kernel_source_sha()
    text = (tree / name).read_text()
    (tree / name).write_text("// a comment\n" + text)
    assert bench.kernel_source_sha() == before
    (tree / name).write_text(text + "\nint changed;\n")
    assert bench.kernel_source_sha() != before
    os.remove(tree / name)
    assert bench.kernel_source_sha() != before
