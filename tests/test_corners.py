"""Vertex corners of a tet mesh (csrc/emu_corners.h), compiled here with g++."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2006_08821_gb300", "csrc")


def test_corner_indices_hold_every_accepted_mesh(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "corners")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "corners_harness.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([exe]).returncode == 0
