"""The order in which a push adds in FP32 is part of its result: a Ritz vector's amplitude magnifies a change of
H-bar by the eigenvectors' condition (11 to 89 for the 2-D waves), so a different order of the same sums
moves it by up to 2e-5.  The values of golden/push_order.json are those of the documented order (the stages
of a pass first to last, two CTAs per SM; row sums and column dots as in pass_ws.cuh, pass_fused.cuh, pass.cuh and lag*.cuh) on
a GB300's 152 SMs, for inputs that are the same on every machine.  The basis is compared bit for bit (a sum
of the bit patterns of every column), H-bar's subdiagonal and beta's last column to 1e-12, which
leaves room for the order of the FP64 sums."""
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "push_order.json")
#            dtype, n, N, reorth, form: stages of 16 tiles and more down to one, several stages a CTA
CASES = {"f32": ("f32", 400001, 140, 1, 0), "bf16": ("bf16", 400001, 150, 1, 0),
         "f32_qr": ("f32", 100003, 70, 1, 1), "f32_cgs1": ("f32", 100003, 70, 0, 0),
         "f32_two_pass": ("f32", 400001, 140, 2, 0), "bf16_two_pass": ("bf16", 100003, 70, 2, 0)}


# dtype, n, N, block: the Cholesky QR of a block works in FP64 up to the rounding of Q to storage
BLOCKS = {"f32_block4": ("f32", 100000, 69, 4), "f32_block2": ("f32", 40000, 41, 2), "bf16_block4": ("bf16", 40000, 41, 4)}


def snapshot_rows(n, N):
    """x_0 noise, x_t = 7/8 x_{t-1} + noise, in FP32: integer arithmetic and separately rounded operations."""
    i = np.arange(n, dtype=np.uint64)
    x = np.zeros(n, dtype=np.float32)
    for t in range(N):
        k = (i + np.uint64(t * n + 1)) * np.uint64(6364136223846793005)
        k ^= k >> np.uint64(29)
        k *= np.uint64(0xBF58476D1CE4E5B9)
        x = x * np.float32(0.875) + ((k >> np.uint64(48)).astype(np.float32) - np.float32(32767.5)) * np.float32(2.0 ** -16)
        yield x


def record(F, dt, n, N, reorth, form):
    import torch
    g = F.FoaDMD(n, N, dt, reorth=reorth, form=form)
    td = {"f32": torch.float32, "bf16": torch.bfloat16}[dt]
    for x in snapshot_rows(n, N):
        st, info = g.push(torch.from_numpy(x).cuda().to(td))
        assert st == 0, info
    return result(g, dt, N)


def record_block(F, dt, n, N, block):
    import torch
    g = F.FoaDMD(n, N, dt)
    X = torch.from_numpy(np.stack(list(snapshot_rows(n, N)))).cuda().to({"f32": torch.float32, "bf16": torch.bfloat16}[dt])
    st, infos = g.push_block(X, block)
    assert st == 0, infos
    return result(g, dt, N)


def result(g, dt, N):
    import torch
    q, _, H, B = g.state()
    assert q == N
    V = g.basis(0, N).contiguous()
    bits = V.view(torch.int32 if dt == "f32" else torch.int16).to(torch.int64).sum(dim=1).cpu().tolist()
    sub = [float(H[c + 1, c]) for c in range(N - 1)]
    g.close()
    return {"bits": bits, "sub": sub, "last": [float(v) for v in B[:N, N - 1]]}


@pytest.mark.parametrize("name", sorted(CASES) + sorted(BLOCKS))
def test_order_of_the_sums(name):
    import torch
    from paper_1805_05821_gb300 import build, foa_dmd
    build.build()
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the stages are dealt over 152 SMs")
    want = json.load(open(GOLDEN))[name]
    got = record(foa_dmd, *CASES[name]) if name in CASES else record_block(foa_dmd, *BLOCKS[name])
    bad = [c for c in range(len(want["bits"])) if want["bits"][c] != got["bits"][c]]
    for key in ("sub", "last"):
        w, g = np.array(want[key]), np.array(got[key])
        assert np.abs(g - w).max() <= 1e-12 * np.abs(w).max(), (key, np.abs(g - w).max())
    assert not bad, f"columns {bad[:8]} of {len(want['bits'])} differ in their bits"


@pytest.mark.parametrize("block", [2, 4])
def test_block_of_tiny_values(block):
    """A block whose R^-1 lies beyond FP32 (entries of about 1e-40): its columns are as orthonormal as entries
    with steps of 2^-149 allow, 2^-149 / 1e-40 = 1.4e-5 each, twice over 64 rows and the three passes."""
    import torch
    from paper_1805_05821_gb300 import build, foa_dmd
    build.build()
    n = 64
    r = np.random.default_rng(block)
    X = np.concatenate([r.standard_normal((1, n)), 1e-40 * r.standard_normal((block, n))]).astype(np.float32)
    g = foa_dmd.FoaDMD(n, 1 + block, "f32")
    st, infos = g.push_block(torch.from_numpy(X).cuda(), block)
    assert st == 0 and g.state()[0] == 1 + block, infos
    V = g.basis(0, 1 + block).double().cpu().numpy()
    assert np.abs(V @ V.T - np.eye(1 + block)).max() <= 6 * 64 * 2.0 ** -149 / 1e-40
    g.close()
