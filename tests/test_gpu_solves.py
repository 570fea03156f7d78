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


@pytest.mark.parametrize("m", [10, 20, 50, 100])
def test_repeated_eigenvalues_are_given_up_early(m, tmp_path):
    """Five-fold eigenvalues: no value has converged after 8 + min(m, 32) / 8 steps, and no more are taken
    before the QR iteration."""
    from paper_1805_05821_gb300.foa_dmd import foa_dmd_test_eig_path
    g = load_with(matrix("multiple", m, 7 * m), tmp_path / "h.ckpt")
    assert g.eig(0.0)["status"] == 0
    assert foa_dmd_test_eig_path(g.h) == (True, 8 + min(m, 32) // 8)
    g.close()


@pytest.mark.parametrize("m,e", [(128, -160), (40, -160), (128, 160), (128, -100), (128, 40), (128, -40)])
def test_scale_decides_without_a_step(m, e, tmp_path):
    """Entries whose scale FP32 cannot hold go to the QR iteration before any step is tried; 2^+-40 does not."""
    from paper_1805_05821_gb300.foa_dmd import foa_dmd_test_eig_path
    H = matrix("waves", m, m)
    g = load_with(np.ldexp(H, e), tmp_path / "h.ckpt")
    res = g.eig(0.0)
    qr, steps = foa_dmd_test_eig_path(g.h)
    assert res["status"] == 0
    assert (qr, steps) == (True, 0) if abs(e) > 60 else (not qr and steps > 0), (qr, steps)
    lam = np.linalg.eigvals(H)
    d = np.abs(np.ldexp(res["lam"].real, -e)[:, None] + 1j * np.ldexp(res["lam"].imag, -e)[:, None] - lam[None, :])
    assert d.min(axis=1).max() <= 64 * m * EPS * np.linalg.norm(H)  # normal to 1e-3: s_i near 1
    g.close()


def hard_matrix(kind, m, seed):
    """Hessenberg matrices whose eigenvalues the simultaneous iteration approaches slowly or at different scales."""
    import scipy.linalg as sl
    g = np.random.default_rng(seed)
    Q = np.linalg.qr(g.standard_normal((m, m)))[0]
    name, val = kind.split(":")
    val = float(val)
    A = np.zeros((m, m))
    ang = np.sort(g.uniform(0.2, 2.9, m // 2))
    if name.startswith("group"):  # one group of 2 or 3 angles, val apart
        c, o = int(name[5:]), m // 6
        ang[o:o + c] = ang[o] + val * np.arange(c)
    if name == "cluster":  # groups of six conjugate pairs on the unit circle, val apart
        ang = np.repeat(ang[::6], 6)[:m // 2] + val * np.tile(np.arange(6), m // 12 + 1)[:m // 2]
    rad = np.ones(m // 2)
    if name == "graded":  # moduli from 1 to 10^-val
        rad = 10.0 ** (-val * np.linspace(0, 1, m // 2))
    for k in range(m // 2):
        c, s = rad[k] * np.cos(ang[k]), rad[k] * np.sin(ang[k])
        A[2 * k:2 * k + 2, 2 * k:2 * k + 2] = [[c, -s], [s, c]]
    if name == "nonnormal":  # far from normal: entries up to val above the diagonal blocks
        A += val * np.triu(g.standard_normal((m, m)), 2) / m
    return np.triu(sl.hessenberg(Q @ A @ Q.T), -1)


@pytest.mark.parametrize("m", [40, 96, 130])
@pytest.mark.parametrize("kind", ["group2:1e-6", "group2:1e-7", "group2:1e-8", "group2:1e-9", "group2:1e-10", "group3:1e-6",
                                  "group3:1e-7", "cluster:1e-4", "cluster:1e-7", "graded:6", "graded:10",
                                  "nonnormal:10", "nonnormal:1000"])
def test_eigenvalues_are_backward_stable(kind, m, tmp_path):
    """Whichever iteration found them, each eigenvalue is one of a matrix within 32 m eps ||H||_F of H: the
    smallest singular value of H - lambda says so directly.  And all are there: matched with LAPACK's,
    they differ by at most that over s_i."""
    import scipy.linalg as sl
    import scipy.optimize as so
    H = hard_matrix(kind, m, m + len(kind))
    g = load_with(H, tmp_path / "h.ckpt")
    res = g.eig(0.0)
    assert res["status"] == 0
    nrm = np.linalg.norm(H)
    back = np.array([np.linalg.svd(H - x * np.eye(m), compute_uv=False)[-1] for x in res["lam"]])
    lam, L, R = sl.eig(H, left=True, right=True)
    s = np.abs(np.sum(L.conj() * R, 0))
    d = np.abs(res["lam"][:, None] - lam[None, :])
    i, j = so.linear_sum_assignment(d)
    from paper_1805_05821_gb300.foa_dmd import foa_dmd_test_eig_path
    print(kind, m, "path", foa_dmd_test_eig_path(g.h), "backward error / (m eps |H|) %.3g" % (back.max() / (m * EPS * nrm)),
          "forward / (m eps |H| / s) %.3g" % (d[i, j] * s[j]).max().__truediv__(m * EPS * nrm), "s %.1e" % s.min())
    g.close()
    assert back.max() <= 32 * m * EPS * nrm
    assert (d[i, j] * s[j]).max() <= 64 * m * EPS * nrm  # LAPACK's own error added
