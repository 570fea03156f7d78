"""Solves whose result used to depend on what a workspace held, or whose spectra decide between the
simultaneous iteration and the QR iteration, on prescribed projected matrices (see test_gpu_roots)."""
import numpy as np
import pytest

from test_gpu_roots import load_with, matrix

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1805_05821_gb300 import build
    build.build()


def low_rank_beta(m, r, seed):
    """Upper triangular, r singular values in [0.1, 1] and the others at 1e-6."""
    g = np.random.default_rng(seed)
    sig = np.concatenate([np.linspace(1.0, 0.1, r), np.full(m - r, 1e-6)])
    X = np.linalg.qr(g.standard_normal((m, m)))[0] * sig
    B = np.linalg.qr(X @ np.linalg.qr(g.standard_normal((m, m)))[0])[1]
    return np.triu(B * np.where(np.diag(B) < 0, -1.0, 1.0)[:, None])


@pytest.mark.parametrize("m,r", [(23, 6), (40, 1), (130, 7)])
def test_more_columns_asked_for_than_the_rank(m, r, tmp_path):
    """n_modes and vec_cols above the truncated rank, as the first solve of a handle: the same as with
    exactly r columns (no column past the rank is looked up in the order)."""
    H, B = matrix("waves", m, m), low_rank_beta(m, r, m + r)
    g = load_with(H, tmp_path / "h.ckpt", beta=B)
    a = g.eig(1e-3, n_modes=m, vec_cols=m)
    h = load_with(H, tmp_path / "h.ckpt", beta=B)
    b = h.eig(1e-3, n_modes=r, vec_cols=r)
    assert a["status"] == b["status"] == 0 and a["r"] == b["r"] == r
    for key in ("lam", "amp", "indicator", "vec", "phi"):
        assert a[key].shape == b[key].shape and np.array_equal(a[key], b[key]), key
    g.close()
    h.close()


@pytest.mark.parametrize("kind,m", [("waves", m) for m in (1, 5, 6, 16, 17, 33, 63, 64, 65, 129, 256, 383, 511)]
                         + [("multiple", 50), ("split", 40), ("scaled", 40)])
def test_which_iteration_found_the_eigenvalues(kind, m, tmp_path):
    """Near-orthogonal matrices of order 6 and more are solved by the simultaneous iteration within
    its 20 FP64 steps; repeated eigenvalues, a zero subdiagonal and entries far outside FP32's range
    are left to the QR iteration."""
    from paper_1805_05821_gb300.foa_dmd import foa_dmd_test_eig_path
    g = load_with(matrix(kind, m, 7 * m + len(kind)), tmp_path / "h.ckpt")
    assert g.eig(0.0)["status"] == 0
    qr, steps = foa_dmd_test_eig_path(g.h)
    if kind == "waves":
        assert qr == (m < 6) and (m < 6 or 0 < steps <= 20), (qr, steps)
    else:
        assert qr
    g.close()
