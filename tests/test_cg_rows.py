"""How many entries of a row the FP32 CG kernels gather at once
(csrc/emu_cgpart.h): the local table decides where there is one, else the row
length. With Jacobi only (degree 1) there is no local table, and the rows of an
irregular mesh have about 14 entries all the same.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2006_08821_gb300", "csrc")


def test_long_rows_are_gathered_wide_without_a_local_table_too(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "rows")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-x", "c++", os.path.join(CSRC, "emu_cgpart.cu"), "-x", "c++",
                    os.path.join(HERE, "cg_rows_harness.cpp"), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    rows = [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    assert rows == [(2, 1, 0, 3, 0), (2, 4, 2, 3, 0), (6, 1, 0, 7, 0), (6, 4, 6, 7, 0),
                    (8, 1, 0, 9, 1), (8, 4, 8, 9, 0), (14, 1, 0, 15, 1), (14, 4, 14, 15, 1)]
