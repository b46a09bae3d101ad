"""The (thread, slot) layout of the capacitance kernel's solving block
(csrc/emu_capslots.h), enumerated on the CPU: every entry of the lower triangle
and of B y is owned once, every address read lies inside the 48 x 48 + 48 sums,
and the slots past the last entry read nothing.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2006_08821_gb300", "csrc")


def test_every_entry_is_owned_once_and_nothing_else_is_read(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "slots")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "cap_slots_harness.cpp"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    tab = np.array([[int(x) for x in line.split()] for line in out.splitlines()])
    assert tab.shape == (1280, 5)
    row, col, src = tab[:, 2], tab[:, 3], tab[:, 4]
    used = col >= 0
    assert used.sum() == 48 * 49 // 2 + 48
    assert len({(r, c) for r, c in zip(row[used], col[used])}) == used.sum()
    assert (col[used] < 48).all() and (row[used] >= col[used]).all() and (row[used] <= 48).all()
    np.testing.assert_array_equal(src[used], np.where(row < 48, 48 * row + col, 2304 + col)[used])
    assert (src[~used] == -1).all(), src[~used].min()
