"""The FP64 reciprocal, reciprocal root, root and Jacobi angle of
csrc/emu_math.cuh, compiled with nvcc through tests/newton_roots_harness.cu.

Between 2^-500 and 2^500 the device takes a third-order step from the
hardware's estimate. That estimate reads the top 20 mantissa bits and returns
20 (PTX manual), so its relative error is below 2^-19. With ulp >= 2^-53 of a
value, the error bounds in ulps follow:
  1/x        remainder e^3 < 2^-57, one rounding:               0.5 + 0.07
  1/sqrt(x)  e rounded in x r (half of 2^-53 in the result), the
             series' remainder 5/16 (2^-18)^3, one rounding:     0.5 + 0.5 + 0.16
  sqrt(x)    a corrected root: the square of the above, one
             rounding:                                           0.5 + 0.01
held to 1, 1.5 and 1 below, against extended precision, and against CUDA's own
expressions within the same bound plus theirs (1, 2 and 0.5 for 1/x, 1/sqrt(x),
sqrt(x) rounded one operation at a time). Outside that range, and for zeros,
subnormals, infinities and NaN, the results are the plain expressions' bits.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2006_08821_gb300", "csrc")
# the range of the third-order steps: the exponent word strictly between these
LO, HI = 2.0**-500, 2.0**500


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


def _values():
    rng = np.random.default_rng(11)
    mid = np.ldexp(rng.uniform(1, 2, 60000), rng.integers(-499, 499, 60000))
    every = np.ldexp(rng.uniform(1, 2, 20000), rng.integers(-1022, 1024, 20000))
    edge = np.array([v * f for v in (LO, HI) for f in (1 - 2.0**-19, 1 - 2.0**-53, 1.0, 1 + 2.0**-52, 1 + 2.0**-21,
                                                       1 + 2.0**-20, 1 + 2.0**-19, 2.0, 0.5)])
    man = np.concatenate([1 + np.arange(64) * 2.0**-52, 2 - np.arange(1, 65) * 2.0**-52, 1 + np.arange(64) * 2.0**-20])
    sub = np.ldexp(rng.integers(1, 1 << 52, 2000).astype(np.float64), -1074)
    special = np.array([0.0, 5e-324, 2.0**-1022, np.finfo(float).max, np.inf, np.nan])
    x = np.concatenate([mid, every, edge, man, sub, special])
    return np.concatenate([x, -x])


@pytest.mark.gpu
def test_roots_against_cuda_and_extended_precision(run):
    x = _values()
    (inv, rs, sq, inv0, rs0, sq0), t = run("device", x, _angles())
    _check_angles(t)
    a = np.abs(x)
    with np.errstate(invalid="ignore"):
        mid = (a > LO * (1 + 2.0**-19)) & (a < HI * (1 - 2.0**-19))
        off = ~((a >= LO) & (a <= HI))
    for got, plain, ok in ((inv, inv0, mid), (rs, rs0, mid & (x > 0)), (sq, sq0, mid & (x > 0))):
        same = (got.view(np.int64) == plain.view(np.int64)) | (np.isnan(got) & np.isnan(plain))
        assert same[off].all(), x[off & ~same]
        assert np.isnan(got[(x < 0) & ~ok & mid]).all()
    L = np.longdouble
    with np.errstate(all="ignore"):
        exact = (1 / L(1) / x.astype(L), 1 / np.sqrt(x.astype(L)), np.sqrt(x.astype(L)))
    assert np.finfo(L).nmant >= 63
    for got, plain, ref, ok, bound, theirs in ((inv, inv0, exact[0], mid, 1.0, 1.0), (rs, rs0, exact[1], mid & (x > 0), 1.5, 2.0),
                                               (sq, sq0, exact[2], mid & (x > 0), 1.0, 0.5)):
        ulp = np.spacing(np.abs(ref[ok].astype(np.float64)))
        err = np.abs(got[ok].astype(L) - ref[ok]) / ulp
        dif = np.abs(got[ok] - plain[ok]) / ulp
        print("max error", float(err.max()), "against CUDA", float(dif.max()), "CUDA's own",
              float((np.abs(plain[ok].astype(L) - ref[ok]) / ulp).max()))
        assert err.max() <= bound, (x[ok][err.argmax()], err.max())
        assert dif.max() <= bound + theirs
