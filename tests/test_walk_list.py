"""The walk's interaction list (csrc/walk_list.cuh) with its lanes run one after another between barriers, on the
host: sums of full chunks, the move of the rest, and the slots of a window's entries."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1610_07279_gb300", "csrc")


def test_list_with_lanes_in_turn(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "walk_list_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, os.path.join(HERE, "walk_list_check.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
