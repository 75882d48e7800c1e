"""Host-side check of the far-field workspace (csrc/farfield_plan.h): the blocks
of directions of one call share one plan, and no count of directions up to the
plan's makes a launch write past its region.  (A plan of its own for the last
block could ask for more row groups, and for up to 231,168 bytes more, than the
full block's: 8,175 directions on 40^3 cells.)"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_block_of_directions_passes_its_workspace(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "farfield_plan_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_0704_0037_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "farfield_plan_check.cpp"), "-o", exe],
                   check=True, capture_output=True)
    rows = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    rows = [r.split() for r in rows if r]
    assert len(rows) == 11 * 5
    for lat, sms, over, big, ok in rows:
        assert int(over) == 0 and int(big) == 0 and ok == "1", (lat, sms, over, big, ok)
