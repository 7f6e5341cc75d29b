"""The DRAM traffic that bench.py reports from a stored capture is dropped when the kernel's source changes."""

import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_1206_0675_gb300", "csrc")


@pytest.mark.parametrize("name", [None, "lgf_common.cuh", "lgf_fixed.cuh"])
def test_stored_traffic_follows_the_source(tmp_path, monkeypatch, name):
    os.makedirs(tmp_path / CSRC)
    for f in ("lgf_site.cu", "lgf_common.cuh", "lgf_fixed.cuh"):
        shutil.copy(os.path.join(bench.ROOT, CSRC, f), tmp_path / CSRC / f)
    key = bench.kernel_source_sha("update_fx")
    monkeypatch.setitem(bench.NCU_TRAFFIC, "update", {**bench.NCU_TRAFFIC["update"], "sha": key, "bytes": 1.0})
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    if name:
        with open(tmp_path / CSRC / name, "a") as f:
            f.write("// changed\n")
    assert bench.ncu_traffic("update") == (None if name else 1.0)
