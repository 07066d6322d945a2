"""Cached tuning choices are tied to every source that they depend on (host logic)."""
import os
import shutil

import pytest

from paper_2301_13601_gb300 import autotune

CSRC = os.path.join(os.path.dirname(os.path.abspath(autotune.__file__)), "csrc")


@pytest.mark.parametrize("name", ["qla_march.cuh", "qla_march.cu", "qla_march_f32_k2.cu", "qla_batch.cu", "qla_api.cu",
                                  "qla_internal.h", "qla_sweep.cuh", "qla_sweep_f32.cu"])
def test_a_changed_source_changes_the_key(tmp_path, name):
    copy = tmp_path / "csrc"
    shutil.copytree(CSRC, copy)
    before = autotune.kernel_version(str(copy))
    assert before == autotune.kernel_version()
    with open(copy / name, "a") as f:
        f.write("// another rule\n")
    assert autotune.kernel_version(str(copy)) != before
