"""The stamp of bench.py's stored sweep counters changes with every file that
decides what a sweep launch does (no GPU needed)."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("name", ["sweep_kernel.cuh", "geometry.cuh", "kernels.cuh", "capi.cu"])
def test_stamp_covers(tmp_path, monkeypatch, name):
    monkeypatch.syspath_prepend(ROOT)
    import bench
    csrc = os.path.join("paper_2605_25872_gb300", "csrc")
    shutil.copytree(os.path.join(ROOT, csrc), tmp_path / csrc)
    before = bench.kernel_version()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_version() == before
    with open(tmp_path / csrc / name, "a") as f:
        f.write("// changed\n")
    assert bench.kernel_version() != before
