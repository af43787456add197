"""The hash under which committed traffic figures count as valid covers every
source the fused stage kernel is compiled from: a change in any of them, the
fixed-point header among them, changes it."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2012_02925_gb300", "csrc")
HEADERS = ["fv_stage.cuh", "fv_face.cuh", "fv_arith.cuh", "fv_fixed.cuh", "fv_viscface.cuh", "fv_internal.h"]


def test_sources_are_the_units_and_their_headers():
    src = bench.kernel_sources()
    assert set(HEADERS) <= set(src)
    assert sum(f.endswith(".cu") for f in src) == 24


@pytest.mark.parametrize("name", HEADERS + ["fv_stage_fp64.cu"])
def test_a_changed_source_changes_the_hash(name, tmp_path, monkeypatch):
    shutil.copytree(os.path.join(bench.ROOT, CSRC), tmp_path / CSRC)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.kernel_hash()
    with open(tmp_path / CSRC / name, "a") as f:
        f.write("// changed\n")
    assert bench.kernel_hash() != before
