"""The guard of bench.py's measured DRAM traffic (CPU): a change to any file that is compiled into the
captured kernels makes the figure null, and it is reported for the captured form of the column pass only."""
import os
import shutil

import pytest

import bench


@pytest.mark.parametrize("name", ["colpass.cu", "passA.cu", "fft.cuh", "common.cuh", "kernels.h", "colteam.cuh", "reduce.cuh",
                                  "df64.cuh"])
def test_every_source_of_the_captured_kernels_is_hashed(tmp_path, monkeypatch, name):
    rel = os.path.join("paper_2006_08303_gb300", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, rel), tmp_path / rel)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_sources_hash()
    with open(tmp_path / rel / name, "a") as f:
        f.write("// changed\n")
    assert bench.kernel_sources_hash() != before


def test_traffic_belongs_to_the_captured_form(monkeypatch):
    monkeypatch.setattr(bench, "TRAFFIC_CAPTURE", {"sources": bench.kernel_sources_hash(),
                                                   "bytes": {"column_pass": 2.0, "prior_pass": 3.0}})
    assert bench.measured_traffic("column_pass", "fused") == 2.0
    assert bench.measured_traffic("column_pass", "split") is None
    assert bench.measured_traffic("prior_pass", "split") == 3.0
