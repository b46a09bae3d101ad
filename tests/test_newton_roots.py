"""The Jacobi angle of csrc/emu_math.cuh, compiled with nvcc through
tests/newton_roots_harness.cu.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2006_08821_gb300", "csrc")


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("roots")
    exe = str(d / "harness")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3", "-I", CSRC,
                    os.path.join(HERE, "newton_roots_harness.cu"), "-o", exe], check=True, capture_output=True)

    def go(where, x, p):
        x, p = np.ascontiguousarray(x, np.float64), np.ascontiguousarray(p, np.float64).reshape(-1, 3)
        with open(d / "in", "wb") as f:
            f.write(np.int64(len(x)).tobytes() + x.tobytes() + np.int64(len(p)).tobytes() + p.tobytes())
        subprocess.run([exe, where, str(d / "in"), str(d / "out")], check=True)
        o = np.fromfile(d / "out")
        return o[:6 * len(x)].reshape(6, -1), o[6 * len(x):]

    return go


def _angles():
    """(app, aqq, apq) with a quotient below, inside and above the third-order
    range, among them equal diagonals beside a subnormal entry."""
    rng = np.random.default_rng(3)
    p = rng.normal(size=(4000, 3))
    p[:1000, 2] *= 2.0 ** rng.uniform(-60, 0, 1000)
    special = [(1.0, 1.0, 1e-310), (0.5, 0.5, 5e-324), (1.0, 1.0, 2.0**-1025), (2.0, 1.0, 1e-310), (1.0, 1.0, 1e-160),
               (1e200, 2e200, 1e170), (0.0, 0.0, 1e-310), (0.0, 1e-310, 1e-310)]
    return np.concatenate([p, special])


def _check_angles(t):
    p = _angles()
    with np.errstate(over="ignore"):
        th = (p[:, 1] - p[:, 0]) / (2.0 * p[:, 2])
        ref = np.copysign(1.0 / (np.abs(th) + np.sqrt(th * th + 1.0)), th)
    assert np.isfinite(t).all(), p[~np.isfinite(t)]
    # a handful of roundings (quotient, square, root, sum, reciprocal) of at most 1.5 ulps each
    np.testing.assert_allclose(t, ref, rtol=16 * 2.0**-53, atol=0)


def test_jacobi_angle_on_the_host(run):
    _check_angles(run("host", [1.0], _angles())[1])
