"""A batched stream's result is its own: the same bits whichever streams are advanced with it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1805_05821_gb300 import build
    build.build()


def advance(F, xs, dt, rounds):
    """Push xs[s][r] in round r for every stream, as long as it has snapshots; states and bases."""
    import torch
    opts = F.foa_dmd_opts_default()
    b = F.foa_dmd_batch_create([x.shape[1] for x in xs], [x.shape[0] for x in xs], dt, opts)
    h = torch.zeros(len(xs), dtype=torch.float64, device="cuda")
    for r in range(rounds):
        p = torch.tensor([x[r].data_ptr() if r < x.shape[0] else 0 for x in xs], dtype=torch.int64, device="cuda")
        F.foa_dmd_batch_push(b, p, h)
        torch.cuda.synchronize()
    out = []
    for s, x in enumerate(xs):
        q, st, H, B = F.foa_dmd_batch_get_state(b, s, x.shape[0])
        V = torch.zeros((x.shape[0], x.shape[1]), dtype=x.dtype, device="cuda")
        F.foa_dmd_batch_get_basis(b, s, 0, q, V, x.shape[1])
        out.append((q, H.copy(), B.copy(), V.float().cpu().numpy()))
    F.foa_dmd_batch_destroy(b)
    return out


@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_company_does_not_change_a_stream(dt):
    """Two streams alone, one by one, and with six larger ones of which two end early."""
    import torch
    from paper_1805_05821_gb300 import foa_dmd as F
    g = torch.Generator(device="cuda").manual_seed(5)
    td = {"f32": torch.float32, "bf16": torch.bfloat16}[dt]

    def stream(n, N):  # rows of a multiple of 8 elements, so that every snapshot is aligned
        return torch.randn((N, (n + 7) // 8 * 8), generator=g, device="cuda").to(td)

    mine = [stream(300000, 40), stream(7001, 30)]
    others = [stream(900000, N) for N in (40, 40, 40, 40, 12, 5)]
    alone = [advance(F, [x], dt, x.shape[0])[0] for x in mine]
    both = advance(F, mine, dt, 40)
    company = advance(F, mine + others, dt, 40)
    for s in range(2):
        assert alone[s][0] == mine[s].shape[0]
        for got in (both[s], company[s]):
            assert got[0] == alone[s][0]
            for a, b in zip(alone[s][1:], got[1:]):
                assert np.array_equal(a, b)
