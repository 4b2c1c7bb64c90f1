"""The digest that ties the committed DRAM counters to the step kernels' code: a change of code in any file that
they are compiled from voids them, a change of wording does not."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2502_09714_gb300", "csrc")


@pytest.mark.parametrize("name", ["dg_step_kernels.cuh", "dg_predictor.cuh", "dg_faces.cuh", "dg_corrector.cuh",
                                  "dg_planes.cuh", "dg_sparse.cuh", "dg_tc.cuh", "dg_team.h", "dg_internal.h",
                                  "gen/basis_lists.cpp", "dg_reference.cpp", "dg_reference.h"])
def test_every_file_of_the_step_kernels_counts(tmp_path, name):
    csrc = str(tmp_path / "csrc")
    shutil.copytree(CSRC, csrc)
    base = bench._kernel_source_digest(csrc)
    assert base == bench._kernel_source_digest()
    p = os.path.join(csrc, name)
    with open(p, "a") as f:
        f.write("\n// a comment\n/* another */\n")
    assert bench._kernel_source_digest(csrc) == base
    with open(p, "a") as f:
        f.write("constexpr int one_more = 1;\n")
    assert bench._kernel_source_digest(csrc) != base
