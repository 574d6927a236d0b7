"""The committed ncu figure of the tile kernel holds for the code it was taken on, headers included: a
change of code in bc_tile.cu or in any file that it includes takes the figure out of the bench's
report, a change of a comment does not."""
import os
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("name", ["bc_tile.cu", "bc_ff.cuh", "bc_common.cuh", "bc_scan.cuh", "bc_internal.h"])
def test_figure_follows_the_code_of_every_included_file(tmp_path, monkeypatch, name):
    import bench
    csrc = os.path.join("paper_1602_00963_gb300", "csrc")
    for d in (csrc, "profiles", "include"):
        shutil.copytree(os.path.join(ROOT, d), tmp_path / d)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.ncu_traffic(128, 0.0) is not None
    path = tmp_path / csrc / name
    text = path.read_text()
    path.write_text(text + "// a comment\n")
    assert bench.ncu_traffic(128, 0.0) is not None
    path.write_text(text + "static int one_more;\n")
    assert bench.ncu_traffic(128, 0.0) is None
