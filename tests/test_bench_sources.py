"""bench.py reports recorded DRAM traffic only while the sources of the passes are the ones
it was recorded on: a change of any of them has to change their hash."""
import os
import shutil

import pytest

import bench


@pytest.mark.parametrize("name", ["xpass_reg.cuh", "ypass_reg.cuh", "zpass_reg.cuh", "reg_step.cuh",
                                  "fft_reg.cuh", "zpass_wide.cuh", "zpass_pair.cuh", "reduce.cuh",
                                  "matvec_impl.cuh", "dda_ops.h", "matvec_fixed.cu",
                                  "xpass_reg_3.cu"])
def test_a_changed_source_changes_the_hash(tmp_path, monkeypatch, name):
    csrc = os.path.join("paper_1305_6497_gb300", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, csrc), tmp_path / csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench._source_hash()
    with open(tmp_path / csrc / name, "a") as f:
        f.write("// changed\n")
    assert bench._source_hash() != before
