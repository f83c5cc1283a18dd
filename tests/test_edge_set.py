"""The host engine's edge set, compiled as plain C++."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1711_00121_gb300", "csrc")


def test_edge_set_matches_unordered_set(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "edge_set_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, os.path.join(HERE, "edge_set_check.cpp"),
                    "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
