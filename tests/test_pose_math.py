"""The sweep's pose math (quaternion Exp, Log, relative pose, mean update) and
identity message on the host, in both precisions, around the limits of their
series branches and over the range of message strengths, against scipy's matrix
exponential / logarithm and the dense Schur complement."""
import os
import shutil
import subprocess

import numpy as np
import pytest
from scipy.linalg import expm
from scipy.spatial.transform import Rotation

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2606_03989_gb300", "csrc")
EPS = {32: 6e-8, 64: 1.2e-16}
# the series end at |theta| = 0.3 (Exp) and sin^2(theta/2) = 0.0223 (Log)
ANGLES = [0.0, 1e-6, 1e-3, 0.1, 0.29, 0.2995, 0.2998, 0.2999, 0.3001, 0.31, 0.6, 1.5, 2.8]


@pytest.fixture(scope="module")
def binary(tmp_path_factory):
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("pose_math") / "pose_math")
    res = subprocess.run([exe, "-x", "cu", "-O2", "-std=c++17", "-I", CSRC, "-o", out,
                          os.path.join(HERE, "math_host", "pose_math.cu")], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-4000:]
    return out


def run(binary, prec, what, cases, n_out):
    cases = np.ascontiguousarray(cases)
    if prec == 32:
        cases = cases.astype(np.float32).astype(np.float64)
    res = subprocess.run([binary, str(prec), what], input=cases.tobytes(), capture_output=True, timeout=300)
    assert res.returncode == 0
    return cases, np.frombuffer(res.stdout).reshape(len(cases), n_out)


def hat(xi):
    w, r = xi[:3], xi[3:]
    return np.array([[0, -w[2], w[1], r[0]], [w[2], 0, -w[0], r[1]], [-w[1], w[0], 0, r[2]], [0, 0, 0, 0]])


def log(T):
    th = Rotation.from_matrix(T[:3, :3]).as_rotvec()
    V = np.zeros((3, 3))
    W = hat(np.r_[th, 0, 0, 0])[:3, :3]
    term = np.eye(3)
    for k in range(1, 40):  # V = sum_k W^(k - 1) / k!
        V += term
        term = term @ W / (k + 1)
    return np.r_[th, np.linalg.solve(V, T[:3, 3])]


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("angle", ANGLES)
def test_poses(binary, prec, angle):
    """Rounding: about 30 operations on values of order 1, and a logarithm's
    conditioning 1 / (pi - angle); 100 eps of that."""
    rng = np.random.default_rng(int(angle * 1e6))
    cases = []
    for _ in range(8):
        a, b = rng.normal(size=6), rng.normal(size=6)
        a[:3] *= min(angle, 0.2) / np.linalg.norm(a[:3])
        b[:3] *= angle / np.linalg.norm(b[:3])
        cases.append(np.r_[a, b])
    cases, out = run(binary, prec, "pose", np.stack(cases), 30)
    tol = 100 * EPS[prec] * (1 + 1 / (np.pi - angle - 0.2))
    for c, o in zip(cases, out):
        Tj, Ti = expm(hat(c[:6])), expm(hat(c[6:]))
        assert np.abs(o[:9].reshape(3, 3) - Ti[:3, :3]).max() < tol
        assert np.abs(o[9:12] - Ti[:3, 3]).max() < tol * 3
        assert np.abs(o[12:18] - c[6:]).max() < tol * 3
        assert np.abs(o[18:24] - log(np.linalg.inv(Tj) @ Ti)).max() < tol * 6
        assert np.abs(o[24:30] - log(Ti @ Tj)).max() < tol * 6


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n_msgs", [0, 1, 3, 7])
@pytest.mark.parametrize("u2", [0.0, 1e-2, 1e4])
def test_identity_message(binary, prec, n_msgs, u2):
    """W = prior + up to seven messages of at most lam each (eigenvalues down to
    1e-4 lam), with and without a photometric rank-one part. The reference subtracts
    lam^2 C^-1 from lam, losing lam / |Lambda| of its FP64 digits."""
    lam, prior = 6.25e6, 400.0
    rng = np.random.default_rng(17 * n_msgs + prec)
    low = np.tril_indices(6)
    cases = []
    for _ in range(40):
        W = prior * np.eye(6)
        for _ in range(n_msgs):
            Q, _ = np.linalg.qr(rng.normal(size=(6, 6)))
            W = W + (Q * (lam * 10 ** rng.uniform(-4, 0, 6))) @ Q.T
        cases.append(np.r_[W[low], rng.normal(size=6) * np.sqrt(u2 * lam), rng.normal(size=6) * lam * 1e-3,
                           rng.normal(size=6) * 1e-3, lam])
    cases, out = run(binary, prec, "message", np.stack(cases), 49)
    for c, o in zip(cases, out):
        W = np.zeros((6, 6))
        W[low] = c[:21]
        W = W + np.tril(W, -1).T
        u, ev, r = c[21:27], c[27:33], c[33:39]
        Ainv = np.linalg.inv(W + lam * np.eye(6))
        z = Ainv @ u
        Ci = Ainv - np.outer(z, z) / (1 + u @ z)
        L = lam * Ainv @ W + lam ** 2 / (1 + u @ z) * np.outer(z, z)
        h = Ainv @ (ev - W @ r)
        e = lam * (h - z * (u @ r + u @ h) / (1 + u @ z))
        assert o[48] == 1
        assert np.linalg.norm(o[:21] - L[low]) < 24 * EPS[prec] * np.linalg.norm(L)
        # eta: the terms that cancel in it
        scale = np.linalg.norm(lam * np.abs(Ainv) @ (np.abs(ev) + np.abs(W) @ np.abs(r))) + \
            lam * np.linalg.norm(z) * np.sum(np.abs(u) * (np.abs(r) + np.abs(Ainv) @ np.abs(ev))) / (1 + u @ z)
        assert np.linalg.norm(o[21:27] - e) < 24 * EPS[prec] * scale
        assert np.linalg.norm(o[27:48] - Ci[low]) < 24 * EPS[prec] * np.linalg.norm(Ci)


def test_a_pivot_that_is_not_positive_is_reported(binary):
    bad = np.r_[np.diag([-2.0, 1, 1, 1, 1, 1])[np.tril_indices(6)], np.zeros(18), 1.0]
    for prec in (32, 64):
        _, out = run(binary, prec, "message", bad[None], 49)
        assert out[0, 48] == 0 and np.isfinite(out).all()
