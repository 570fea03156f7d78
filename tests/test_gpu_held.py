"""Edges of the register-held passes (stages of 1 to 16 tiles), of the FP64 stages and of the block push's
two Cholesky paths, against the FP64 oracle on the same storage-rounded inputs.  Tolerances as in
test_gpu_push (column by column within C u_s kappa_2(X_{1:p}) <= 1e-2, FP64 1e-10 normwise)."""
import numpy as np
import pytest

from gpu_util import PARITY_C, U, compare_state, gaussian, run_gpu, to_device
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1805_05821_gb300 import build
    build.build()


@pytest.mark.parametrize("dt", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("reorth", [1, 2])
@pytest.mark.parametrize("n,N", [(160, 20), (513, 34), (1541, 70), (8193, 136)])
def test_stage_edges(dt, reorth, n, N):
    """j runs over every stage size (16 tiles at j = 1 to one), with a ragged last tile and a last stage
    that is partly empty."""
    Xr, Xd = to_device(gaussian(n, N, 7 * n + N), dt)
    g, infos = run_gpu(Xd, n, N, dt, reorth=reorth)
    assert all(st == 0 for st, _ in infos)
    o = oracle.FoaOracle(n, N, storage=dt, reorth=reorth)
    for t in range(N):
        assert o.push(Xr[:, t])[0] == "ok"
    compare_state(g, o, dt, with_basis=True, label=f"{dt} reorth {reorth} n={n}")


@pytest.mark.parametrize("block", [2, 4])
@pytest.mark.parametrize("delta", [1.0, 1e-2, 5e-4])
def test_block_conditions(block, delta):
    """Blocks whose snapshots differ by delta: R1's condition number is about 1/delta, on both sides of
    the bound (512) under which one Cholesky step is taken.  beta's and V's columns by the law; the
    H-bar columns, whose error the QR form amplifies beyond it at 1/delta = 2000, by the relation that
    defines them, beta_{:,2:} = H-bar beta, to the rounding of a forward substitution of N terms."""
    from paper_1805_05821_gb300.foa_dmd import FoaDMD
    n, N = 6000, 1 + 3 * block
    g0 = np.random.default_rng(int(1e6 * delta) + block)
    X = g0.standard_normal((n, N))
    for s in range(1, N, block):
        for k in range(1, block):
            X[:, s + k] = X[:, s] + delta * X[:, s + k]
    Xr, Xd = to_device(X, "f32")
    g = FoaDMD(n, N, "f32", breakdown_tol=1e-12)
    st, infos = g.push_block(Xd, block=block)
    assert st == 0, infos
    o = oracle.FoaOracle(n, N, breakdown_tol=1e-12, storage="f32", form="qr")
    o.push(Xr[:, 0])
    for s in range(1, N, block):
        o.push_block(Xr[:, s:s + block])
    q, _, H, B = g.state()
    assert q == o.q == N
    bound = PARITY_C["f32"] * U["f32"] * np.linalg.cond(Xr)
    assert bound <= 1e-2
    assert (np.linalg.norm(B - o.B, axis=0) <= bound * np.linalg.norm(o.B, axis=0)).all()
    V = g.basis(0, N).double().cpu().numpy()
    Vo = np.linalg.solve(o.B.T, Xr.T)  # V = X beta^-1
    assert (np.linalg.norm(V - Vo, axis=1) <= bound).all()
    res = np.abs(B[:, 1:] - H[:, :N - 1] @ B[:N - 1, :N - 1])
    assert (res[:, :] <= 4 * N * 2.0 ** -53 * (np.abs(H[:, :N - 1]) @ np.abs(B[:N - 1, :N - 1])) + 1e-300).all()
