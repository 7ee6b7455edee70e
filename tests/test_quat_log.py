"""The pose Log on quaternions of either sign: q and -q are one rotation, and a
product of two poses of nearly half a turn each has w < 0 (compiled for the host)."""
import os
import shutil
import subprocess

import numpy as np
import pytest
from scipy.linalg import expm

from test_pose_math import CSRC, EPS, HERE, hat, log


@pytest.fixture(scope="module")
def binary(tmp_path_factory):
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("quat_log") / "quat_log")
    res = subprocess.run([exe, "-x", "cu", "-O2", "-std=c++17", "-I", CSRC, "-o", out,
                          os.path.join(HERE, "math_host", "quat_log.cu")], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    return out


def run(binary, prec, what, cases):
    res = subprocess.run([binary, str(prec), what], input=np.ascontiguousarray(cases).tobytes(), capture_output=True,
                         timeout=300)
    assert res.returncode == 0
    return np.frombuffer(res.stdout).reshape(len(cases), 6)


@pytest.mark.parametrize("prec", [32, 64])
def test_a_quaternion_and_its_negative_have_the_same_log(binary, prec):
    rng = np.random.default_rng(3)
    cases = []
    for half in (0.0, 1e-30, 1e-23, 1e-8, 1e-3, 0.1, 0.149, 0.151, 0.8, 1.5):  # half angles; the series end at 0.15
        n = rng.normal(size=3)
        cases.append(np.r_[np.cos(half), np.sin(half) * n / np.linalg.norm(n), rng.normal(size=3)])
    cases = np.stack(cases)
    if prec == 32:
        cases = cases.astype(np.float32).astype(np.float64)
    neg = cases * np.r_[-np.ones(4), np.ones(3)]
    a, b = run(binary, prec, "log", cases), run(binary, prec, "log", neg)
    assert np.isfinite(b).all()
    assert np.array_equal(a, b)
    assert np.array_equal(b[0], np.r_[np.zeros(3), cases[0, 4:]])  # (-1, 0, 0, 0): no rotation


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("gap", [0.0, 1e-6, 1e-3, 0.05, 0.2])
def test_relative_pose_of_opposite_rotations_near_half_a_turn(binary, prec, gap):
    """Rounding as in the other poses: 600 eps of values up to |t| of 4 (both poses'
    translations, about 30 operations each)."""
    rng = np.random.default_rng(int(gap * 1e6))
    cases = []
    for axis in list(np.eye(3)) + [n / np.linalg.norm(n) for n in rng.normal(size=(5, 3))]:
        cases.append(np.r_[axis * (np.pi - gap), rng.normal(size=3), -axis * (np.pi - gap), rng.normal(size=3)])
    cases = np.stack(cases)
    if prec == 32:
        cases = cases.astype(np.float32).astype(np.float64)
    out = run(binary, prec, "between", cases)
    for c, o in zip(cases, out):
        ref = log(np.linalg.inv(expm(hat(c[:6]))) @ expm(hat(c[6:])))
        assert np.abs(o - ref).max() < 600 * EPS[prec] * 4
