"""The identity message of a coupling much weaker than what the sender knows (a strong
pose prior, or a large sigma_R): W far above lam, where Lambda approaches lam I and its
off-diagonal entries are of order lam^2 / W. On the host, in both precisions."""
import numpy as np
import pytest

from test_pose_math import EPS, binary, run  # noqa: F401  (binary is a fixture)


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("ratio", [1e1, 1e3, 1e6, 1e9])
@pytest.mark.parametrize("u2", [0.0, 1.0, 1e4])
def test_weak_coupling(binary, prec, ratio, u2):  # noqa: F811
    """W = ratio lam I + three messages of at most lam each, so A = W + lam I has a
    condition number below 2 and the bounds are those of rounding: 24 eps of each
    result's norm (about 20 operations an entry, in random directions)."""
    lam = 6.25e6
    rng = np.random.default_rng(int(np.log10(ratio)) + prec)
    low = np.tril_indices(6)
    cases = []
    for _ in range(40):
        W = ratio * lam * np.eye(6)
        for _ in range(3):
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
        L = lam * np.eye(6) - lam ** 2 * Ci  # lam C^-1 V; no cancellation where V is far above lam
        h = Ainv @ (ev - W @ r)
        e = lam * (h - z * (u @ r + u @ h) / (1 + u @ z))
        assert o[48] == 1
        assert np.linalg.norm(o[:21] - L[low]) < 24 * EPS[prec] * np.linalg.norm(L)
        off = np.array([i != j for i, j in zip(*low)])  # the off-diagonal entries by themselves
        assert np.abs(o[:21] - L[low])[off].max() < 24 * EPS[prec] * lam ** 2 * np.abs(Ci).max()
        scale = np.linalg.norm(lam * np.abs(Ainv) @ (np.abs(ev) + np.abs(W) @ np.abs(r))) + \
            lam * np.linalg.norm(z) * np.sum(np.abs(u) * (np.abs(r) + np.abs(Ainv) @ np.abs(ev))) / (1 + u @ z)
        assert np.linalg.norm(o[21:27] - e) < 24 * EPS[prec] * scale
        assert np.linalg.norm(o[27:48] - Ci[low]) < 24 * EPS[prec] * np.linalg.norm(Ci)
