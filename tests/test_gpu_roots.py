"""Eigenvalues by simultaneous iteration, the QR iteration that takes over from it, and the Jacobi SVD
of the rank truncation, on prescribed projected matrices (written as a checkpoint and loaded) against
LAPACK.

Tolerances are fixed by first-order perturbation theory: both solvers are backward stable, so an
eigenvalue moves by at most 32 m eps ||H||_F / s_i (s_i the cosine between its left and right
eigenvectors), asserted where that is below 1e-3; the residual of a returned vector is at most
1e3 m eps ||H||_F.
"""
import struct

import numpy as np
import pytest

from gpu_util import match

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1805_05821_gb300 import build
    build.build()


def fnv1a(h, data):
    for b in data:
        h = ((h ^ b) * 1099511628211) & 0xFFFFFFFFFFFFFFFF
    return h


def load_with(H, path, b11=2.0, h_last=0.25, beta=None):
    """A handle whose projected matrix is H (m x m upper Hessenberg), beta = b11 I unless given."""
    from paper_1805_05821_gb300.foa_dmd import FoaDMD
    m = H.shape[0]
    K = m + 1
    f32 = K > 384
    Hb = np.zeros((K, K), order="F")
    Hb[:m, :m] = H
    Hb[m, m - 1] = h_last
    B = np.asfortranarray(np.eye(K) * b11)
    if beta is not None:
        B[:m, :m] = beta
    V = np.zeros(K, dtype=np.float32 if f32 else np.float64)
    body = Hb.tobytes("F") + B.tobytes("F") + V.tobytes()
    head = b"FOADMD1\0" + struct.pack("<iiiiqii", 1, 1 if f32 else 0, K, K, 1, 0, 0)
    head += struct.pack("<Q", fnv1a(1469598103934665603, body))
    with open(path, "wb") as f:
        f.write(head + body)
    return FoaDMD.load(str(path), "f32" if f32 else "f64", 1, K)


def matrix(kind, m, seed):
    import scipy.linalg as sl
    g = np.random.default_rng(seed)
    A = g.standard_normal((m, m))
    if kind == "waves":  # near the unit circle, as undamped waves with noise give it
        A = np.linalg.qr(A)[0] + 1e-3 * g.standard_normal((m, m))
    elif kind == "symmetric":  # a real interval
        A = A + A.T
    elif kind == "multiple":  # every eigenvalue five times
        Q = np.linalg.qr(A)[0]
        A = Q @ np.diag(np.repeat(np.arange(1.0, m // 5 + 1), 5)) @ Q.T
    H = np.triu(sl.hessenberg(A) if m > 2 else A, -1)
    if kind == "split":
        H[m // 2, m // 2 - 1] = 0.0
    if kind == "scaled":
        H *= 1e-120
    return H


@pytest.mark.parametrize("kind,m", [("waves", m) for m in (1, 2, 15, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257, 383, 511)]
                         + [("dense", 48), ("dense", 200), ("symmetric", 60), ("multiple", 50), ("split", 40),
                            ("scaled", 40)])
def test_eigenvalues_and_vectors(kind, m, tmp_path):
    H = matrix(kind, m, 7 * m + len(kind))
    g = load_with(H, tmp_path / "h.ckpt")
    r = g.eig(0.0, vec_cols=m)
    assert r["status"] == 0 and r["r"] == m
    lam, L, R = __import__("scipy.linalg").linalg.eig(H, left=True, right=True)
    s = np.abs(np.sum(L.conj() * R, 0))
    nrm = np.linalg.norm(H)
    d, idx = match(r["lam"], lam)
    bound = 32 * m * EPS * nrm / np.maximum(s, 1e-300)
    ok = bound <= 1e-3 * nrm
    d = np.abs(r["lam"][:, None] - lam[None, :])
    import scipy.optimize as so
    i, j = so.linear_sum_assignment(d)
    assert np.all((d[i, j] <= bound[j]) | ~ok[j]), (d[i, j] / bound[j]).max()
    # conjugate pairs are exact and adjacent, +Im first
    k = 0
    while k < m:
        if r["lam"][k].imag == 0.0:
            k += 1
            continue
        assert r["lam"][k].imag > 0.0 and r["lam"][k + 1] == np.conj(r["lam"][k])
        k += 2
    Z = r["vec"]
    assert np.linalg.norm(H @ Z - Z * r["lam"][None, :], axis=0).max() <= 1e3 * m * EPS * nrm
    if kind in ("waves", "dense"):  # amplitudes: Z c = b11 e_1
        e1 = np.zeros(m)
        e1[0] = 2.0
        assert np.linalg.norm(Z @ r["amp"] - e1) <= 1e3 * m * EPS * np.linalg.cond(Z) ** 2
        assert np.allclose(r["indicator"], 0.25 * np.abs(Z[-1]), rtol=0, atol=1e3 * m * EPS)
    g.close()


@pytest.mark.parametrize("m,r,fall", [(1, 1, 0.0), (2, 2, 1.0), (3, 2, 3.0), (64, 40, 4.0), (127, 127, 3.0), (128, 20, 9.0),
                                      (129, 64, 6.0), (256, 100, 5.0), (257, 30, 3.0), (383, 96, 4.0), (511, 60, 5.0)])
def test_truncated_solve(m, r, fall, tmp_path):
    """Singular values and eigenvalues of U_r^T H U_r: beta upper triangular with r singular values
    spread over 10^-fall .. 1 and the others 1e-3 below them.  |d sigma| <= 32 m eps sigma_1, the
    eigenvalues by the bound above with the perturbation of U_r, 32 m eps sigma_1 / (gap)."""
    g = np.random.default_rng(3 * m + r)
    sig = np.concatenate([10.0 ** (-fall * np.linspace(0, 1, r)), np.full(m - r, 10.0 ** (-fall - 3))])
    X = np.linalg.qr(g.standard_normal((m, m)))[0] * sig
    B = np.linalg.qr(X @ np.linalg.qr(g.standard_normal((m, m)))[0])[1]
    B = B * np.where(np.diag(B) < 0, -1.0, 1.0)[:, None]
    H = matrix("waves", m, m + 1)
    tol = 10.0 ** (-fall - 1.5)
    h = load_with(H, tmp_path / "h.ckpt", beta=np.triu(B))
    res = h.eig(tol)
    assert res["status"] == 0 and res["r"] == r, res["r"]
    U, s, _ = np.linalg.svd(np.triu(B))
    assert np.abs(res["sigma"] - s[:r]).max() <= 32 * m * EPS * s[0]
    import scipy.linalg as sl
    import scipy.optimize as so
    G = U[:, :r].T @ H @ U[:, :r]
    lam, L, R = sl.eig(G, left=True, right=True)
    cond = 1.0 / np.abs(np.sum(L.conj() * R, 0))
    gap = s[r - 1] - (s[r] if r < m else 0.0)
    bound = 32 * m * EPS * np.linalg.norm(H, 2) * cond * (1.0 + s[0] / gap)
    d = np.abs(res["lam"][:, None] - lam[None, :])
    i, j = so.linear_sum_assignment(d)
    ok = bound[j] <= 1e-3
    assert np.all((d[i, j] <= bound[j]) | ~ok), (d[i, j] / bound[j]).max()
    h.close()
