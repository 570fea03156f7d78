"""The work that users of this library have it do, as cases that can be timed and compared.

Snapshots are travelling waves on a grid (the structure of the waves and fields workloads of
paper_1805_05821_gb300/synth.py), drawn from the seed with torch: frequencies spread over
(0, pi), amplitudes falling geometrically from 1 to 1/decay, measurement noise.  Two shapes of
data cover what a stream meets:

  waves    as many waves as make the N snapshots linearly independent: every pushed direction is
           signal, every Ritz value is a wave's;
  fields   fewer waves than snapshots and noise below them: the projected matrix is truncated to
           the waves' rank with an explicit rank_tol between signal and noise.

Results of FP32 and BF16 streams are returned as FP32 (their H-bar, beta and Ritz values carry the
storage type's error), results of FP64 streams as FP64.  Modes are returned times their
amplitudes, c_i Phi_i, as they enter a reconstruction: that product does not depend on the phase
and sign conventions of the eigenvectors and of the singular vectors.
"""
import math

import numpy as np
import torch

from paper_1805_05821_gb300 import foa_dmd as F

TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest stream, watched push by push: 32 snapshots of a rank-10 system, the stream
        # breaks down at push 11 (the planted n=4096, N=32 configuration) and is then solved
        {"name": "planted_f64", "kind": "push", "dtype": "f64", "n": 4096, "N": 32, "waves": 5, "noise": 0.0,
         "info": True, "eig": "full"},
        # a short stream on a small grid, every push's result read (sizes of the smoke run)
        {"name": "small_f32", "kind": "push", "dtype": "f32", "n": 16384, "N": 80, "waves": 40, "noise": 1e-3,
         "info": True, "eig": "none"},
        # the plain FP64 form on the 1024 x 1024 grid
        {"name": "waves2d_f64", "kind": "push", "dtype": "f64", "n": 1048576, "N": 96, "waves": 48, "noise": 1e-3,
         "info": False, "eig": "none"},
        # the 1024 x 1024 grid in FP32, N = 200, an indicator every 40 pushes and all Ritz values at the end
        {"name": "waves2d_f32", "kind": "push", "dtype": "f32", "n": 1048576, "N": 200, "waves": 100, "noise": 1e-3,
         "info": False, "eig": "full", "every": 40},
        # a 128^3 grid stored in BF16, snapshots handed over as one block of memory (push_batch)
        {"name": "waves3d_bf16", "kind": "push_batch", "dtype": "bf16", "n": 2097152, "N": 160, "waves": 96,
         "noise": 1e-2, "info": True, "eig": "none"},
        # four fields on a 128^3 grid: long FP32 stream, then truncated Ritz values and 32 modes
        {"name": "fields_f32", "kind": "push", "dtype": "f32", "n": 8388608, "N": 256, "waves": 48, "noise": 1e-2,
         "info": False, "eig": "trunc", "modes": 32},
        # an unstructured mesh (odd number of points) with the two-pass push
        {"name": "mesh_two_pass_f32", "kind": "push", "dtype": "f32", "n": 3500017, "N": 128, "waves": 64,
         "noise": 1e-3, "info": False, "eig": "none", "reorth": 2},
        # snapshots that arrive four at a time
        {"name": "block4_f32", "kind": "push_block", "dtype": "f32", "n": 4194304, "N": 256, "waves": 128,
         "noise": 1e-2, "block": 4, "info": True, "eig": "none"},
        # snapshots that a simulation leaves in pinned host memory, odd length
        {"name": "host_f32", "kind": "push_host", "dtype": "f32", "n": 1000003, "N": 100, "waves": 50, "noise": 1e-3,
         "info": False, "eig": "none"},
        # many uneven streams advanced together under a CUDA graph, from creation to their states
        {"name": "streams_f32", "kind": "streams", "dtype": "f32", "streams": 48, "n_low": 16384, "n_high": 1048576,
         "N_low": 50, "N_high": 120, "sizes_seed": 4},
        # the eigensolve by itself, all Ritz values of a 255 x 255 projected matrix in FP64
        {"name": "eig_full_f64", "kind": "eig", "dtype": "f64", "n": 16384, "N": 256, "waves": 128, "noise": 1e-3,
         "eig": "full", "vectors": 16},
        # the truncated eigensolve by itself at the fields configuration's m = 383 (r = 96), with 32 modes
        {"name": "eig_trunc_f32", "kind": "eig", "dtype": "f32", "n": 1048576, "N": 384, "waves": 48, "noise": 1e-2,
         "eig": "trunc", "modes": 32},
    ]


def draw(rng):
    def size(lo, hi):
        v = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
        return v | 1 if rng.random() < 0.5 else v

    kind = rng.choice(["push", "push", "push", "push_batch", "push_block", "push_host", "streams", "eig", "eig"])
    if kind == "streams":
        low = size(4000, 60000)
        return {"kind": kind, "dtype": rng.choice(["f32", "f32", "bf16"]), "streams": rng.randint(3, 56),
                "n_low": low, "n_high": low * rng.randint(4, 16), "N_low": rng.randint(8, 40),
                "N_high": rng.randint(41, 120), "sizes_seed": rng.randint(1, 10 ** 6)}
    if kind == "eig":
        trunc = rng.random() < 0.5
        N, dtype = min(384, size(24, 384)), rng.choice(["f64", "f32"])
        c = {"kind": kind, "dtype": dtype, "n": size(8192, 40000 if dtype == "f64" else 400000), "N": N,
             "waves": max(2, N // 8) if trunc else (N + 1) // 2, "noise": 1e-2 if trunc else 1e-3,
             "eig": "trunc" if trunc else "full"}
        if trunc:
            c["modes"] = rng.choice([0, 8, 32])
        else:
            c["vectors"] = rng.choice([0, 8])
        return c
    dtype = rng.choice(["f32", "bf16"]) if kind == "push_block" else rng.choice(["f32", "f32", "f32", "f64", "bf16"])
    N = size(12, 256)
    most = {"f64": 6e9, "f32": 1.2e11, "bf16": 1.2e11}[dtype] / N / N  # no dearer than the largest listed ones
    n = size(3000, max(6000, min(8388608, most)))
    c = {"kind": kind, "dtype": dtype, "n": max(n, 16 * N), "N": N, "waves": (N + 1) // 2 + rng.randint(0, N // 4),
         "noise": 1e-2 if dtype == "bf16" or kind == "push_block" else 1e-3, "info": rng.random() < 0.5, "eig": "none"}
    if kind == "push_block":
        c["block"] = rng.choice([2, 4])
    elif kind == "push":
        form = rng.choice(["default", "default", "two_pass", "qr"])
        if form == "two_pass":
            c["reorth"] = 2
        elif form == "qr":
            c["form"] = 1
    return c


# ----------------------------------------------------------------------------------- inputs
DECAY = 10.0  # amplitudes fall from 1 to 1/DECAY
RANK_TOL = 2e-2  # between the weakest wave and the noise of the fields data


def snapshots(n, N, waves, noise, seed, dtype):
    """N snapshots (rows, leading dimension padded to 16 bytes) of `waves` travelling waves on n points."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    per = 16 // SIZE[dtype]
    ld = (n + per - 1) // per * per
    X = torch.zeros((N, ld), dtype=TORCH[dtype], device="cuda")
    work = torch.float64 if dtype == "f64" else torch.float32
    m = torch.arange(waves, device="cuda", dtype=torch.float64)
    u = torch.rand((2, waves), generator=g, device="cuda", dtype=torch.float64)
    omega = math.pi * (m + 0.35 + 0.3 * u[0]) / waves
    amp = DECAY ** (-m[torch.randperm(waves, generator=g, device="cuda")] / max(1, waves - 1))
    t = torch.arange(N, device="cuda", dtype=torch.float64)
    # x_t = sum_m a_m cos(k_m . r + phi_m - omega_m t): cosine and sine tables in space and time
    T = torch.cat([amp * torch.cos(t[:, None] * omega), amp * torch.sin(t[:, None] * omega)], 1).to(work)
    side = max(2, int(math.sqrt(n)))
    most = min(64, side // 2 - 1)  # wave numbers the grid resolves, no two waves with the same one
    cell = torch.randperm(most * most, generator=g, device="cuda")[:waves]
    k1, k2 = (1 + cell % most).to(torch.float32), (cell // most).to(torch.float32)
    phi = (2 * math.pi * u[1]).to(torch.float32)
    rms = float(torch.sqrt((amp ** 2).sum() / 2))
    chunk = max(4096, (1 << 26) // max(1, 2 * waves))
    for r0 in range(0, n, chunk):
        r = torch.arange(r0, min(n, r0 + chunk), device="cuda")
        a, b = (r % side).to(torch.float32) / side, (r // side).to(torch.float32) / side
        arg = 2 * math.pi * (a[:, None] * k1 + b[:, None] * k2) + phi
        S = torch.cat([torch.cos(arg), torch.sin(arg)], 1).to(work)
        P = T @ S.T
        if noise:
            P += noise * rms * torch.randn(P.shape, generator=g, device="cuda", dtype=work)
        X[:, r0:r0 + P.shape[1]] = P.to(X.dtype)
    return X


def stream_sizes(case):
    rng = np.random.RandomState(case["sizes_seed"])
    n = np.exp(rng.uniform(math.log(case["n_low"]), math.log(case["n_high"]), case["streams"])).astype(int)
    N = rng.randint(case["N_low"], case["N_high"] + 1, case["streams"])
    return [(int(max(a, 16 * b)), int(b)) for a, b in zip(n, N)]


def stream_snapshots(case, seed):
    return [snapshots(n, N, (N + 1) // 2, 1e-2, int(seed) * 1000 + s, case["dtype"])
            for s, (n, N) in enumerate(stream_sizes(case))]


def case_snapshots(case, seed):
    return snapshots(case["n"], case["N"], case["waves"], case["noise"], seed, case["dtype"])


# ----------------------------------------------------------------------------------- one pass
def prepare(case, seed):
    if case["kind"] == "streams":
        xs = stream_snapshots(case, seed)
        rounds = max(x.shape[0] for x in xs)
        # the snapshot each stream pushes in each round, as a table of device pointers (0: none left)
        table = torch.tensor([[int(x[r].data_ptr()) if r < x.shape[0] else 0 for x in xs] for r in range(rounds)],
                             dtype=torch.int64).cuda()
        return {"case": case, "xs": xs, "table": table, "stream": torch.cuda.Stream(),
                "ptrs": torch.zeros(len(xs), dtype=torch.int64, device="cuda"),
                "h_last": torch.zeros(len(xs), dtype=torch.float64, device="cuda")}
    X = case_snapshots(case, seed)
    dmd = F.FoaDMD(case["n"], case["N"], case["dtype"], reorth=case.get("reorth", 1), form=case.get("form", 0),
                   indicator_every=case.get("every", 0))
    s = {"case": case, "X": X, "dmd": dmd}
    if case["kind"] == "push_host":
        s["X"] = X.cpu().pin_memory()
    if case["kind"] == "eig":  # the stream is in the handle already
        st, _ = dmd.push_batch(X)
        assert st == F.OK, st
        s["X"] = None
    if case.get("modes"):
        ld = (case["n"] + 3) // 4 * 4
        s["phi"] = torch.zeros((2 * case["modes"], ld), device="cuda",
                               dtype=torch.float64 if case["dtype"] == "f64" else torch.float32)
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "streams":
        return run_streams(state)
    dmd, X = state["dmd"], state["X"]
    if case["kind"] != "eig":
        dmd.reset()
        push(case, dmd, X)
    out = {}
    if case["kind"] != "eig":
        q, stopped, H, B = dmd.state()
        out["q"] = q
        out["H"], out["B"] = result(case, H), result(case, B)
        if not case.get("modes"):
            out["V"] = dmd.basis(0, q)
    if case.get("every"):
        out["indicators"] = result(case, np.array([v for _, _, v in dmd.indicators()]))
    if case["eig"] != "none":
        out.update(solve(case, dmd, state.get("phi")))
    return out


def push(case, dmd, X):
    N = case["N"]
    if case["kind"] == "push_batch":
        dmd.push_batch(X, case["info"])
    elif case["kind"] == "push_block":
        dmd.push_block(X, case["block"], case["info"])
    elif case["kind"] == "push_host":
        step = X.stride(0) * X.element_size()
        for t in range(N):
            F.foa_dmd_push_host(dmd.h, X.data_ptr() + t * step, case["info"])
    else:
        for t in range(N):
            status, _ = dmd.push(X[t], case["info"])
            if status != F.OK:  # a dependent snapshot ends the stream
                break


def solve(case, dmd, phi):
    nm = case.get("modes", 0)
    res = F.foa_dmd_eig(dmd.h, RANK_TOL if case["eig"] == "trunc" else 0.0, case["N"], nm, phi,
                        phi.shape[1] if nm else 0, case.get("vectors", 0))
    out = {"r": res["r"], "lam": result(case, res["lam"]), "amp": result(case, np.abs(res["amp"])),
           "indicator": result(case, res["indicator"])}
    if case["eig"] == "trunc":
        out["sigma"] = result(case, res["sigma"])
    if case.get("vectors"):
        out["vec"] = result(case, res["vec"] * res["amp"][None, :res["vec"].shape[1]])
    if nm:
        k = min(nm, res["r"])
        c = torch.from_numpy(res["amp"][:k]).to("cuda")
        re, im = phi[0:2 * k:2], phi[1:2 * k:2]
        cr, ci = c.real.to(phi.dtype)[:, None], c.imag.to(phi.dtype)[:, None]
        out["modes_re"] = torch.addcmul(re * cr, im, ci, value=-1)[:, :case["n"]]
        out["modes_im"] = torch.addcmul(re * ci, im, cr)[:, :case["n"]]
    return out


def result(case, a):
    if case["dtype"] == "f64":
        return a
    return a.astype(np.complex64 if np.iscomplexobj(a) else np.float32)


def run_streams(state):
    case, xs, table, stream = state["case"], state["xs"], state["table"], state["stream"]
    opts = F.foa_dmd_opts_default()
    opts.cuda_stream = stream.cuda_stream
    b = F.foa_dmd_batch_create([x for x, _ in stream_sizes(case)], [x.shape[0] for x in xs], case["dtype"], opts)
    graph = torch.cuda.CUDAGraph()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        with torch.cuda.graph(graph, stream=stream):
            F.foa_dmd_batch_push(b, state["ptrs"], state["h_last"])
        for r in range(table.shape[0]):
            state["ptrs"].copy_(table[r])
            graph.replay()
    H, B, q = [], [], []
    for s, x in enumerate(xs):
        qs, _, Hs, Bs = F.foa_dmd_batch_get_state(b, s, x.shape[0])
        q.append(qs)
        H.append(Hs.ravel())
        B.append(Bs.ravel())
    F.foa_dmd_batch_destroy(b)
    return {"q": np.array(q), "H": result(case, np.concatenate(H)), "B": result(case, np.concatenate(B))}


# ----------------------------------------------------------------------------------- its least work
def work(case):
    """Each push (or block of pushes) reads its snapshots and the basis once and writes the new basis
    vectors; five products with the basis: the pre-vector, two projections and their two corrections
    (the QR view and the block push have no pre-vector)."""
    if case["kind"] == "streams":
        pairs = stream_sizes(case)
    else:
        pairs = [(case["n"], case["N"])]
    nbytes = flops = 0.0
    if case["kind"] == "eig":
        m = case["N"] - 1
        r = m if case["eig"] == "full" else min(m, 2 * case["waves"])
        es = 8 if case["dtype"] == "f64" else 4
        nbytes += 2 * 8 * m * m + 8 * 5 * r
        # Ritz values of the r x r matrix (10 r^3, Golub & Van Loan), SVD of the m x m one where truncated
        flops += 10.0 * r ** 3 + (4.0 * m ** 3 + 4.0 * m * m * r if case["eig"] == "trunc" else 0.0)
        if case.get("modes"):
            nbytes += case["n"] * (SIZE[case["dtype"]] * m + 2 * es * case["modes"])
            flops += 4.0 * case["n"] * m * case["modes"]
        return {"bytes": nbytes, "flops": flops}
    block = case.get("block", 1)
    for n, N in pairs:
        steps = 2 * case["waves"] + 1 if case.get("noise") == 0.0 else N  # pushes until the breakdown
        es = SIZE[case["dtype"]]
        pushes = steps * (steps - 1) / 2.0
        products = 4 if case.get("form") or block > 1 else 5
        nbytes += n * es * (pushes / block + 2.0 * steps)
        flops += 2.0 * products * n * pushes
        if case.get("eig") in ("full", "trunc"):
            more = work({**case, "kind": "eig", "N": steps})
            nbytes += more["bytes"]
            flops += more["flops"]
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------------------------- in 64 bits
def qr64(X, n):
    """R (positive diagonal) and Q of the snapshots (rows of X) in 64 bits, Cholesky QR three times."""
    A = X[:, :n].to(torch.float64).T
    R = torch.eye(A.shape[1], dtype=torch.float64, device=A.device)
    for _ in range(3):
        L = torch.linalg.cholesky(A.T @ A)
        A = torch.linalg.solve_triangular(L, A.T, upper=False).T
        R = L.T @ R
    return R, A


def projected(X, n, rank=None):
    """beta, H-bar (square, zero past the last column) and the basis of a whole stream, from its QR factors."""
    N = X.shape[0]
    steps = N if rank is None else rank
    R, Q = qr64(X[:steps], n)
    H = np.zeros((N, N))
    B = np.zeros((N, N))
    r = R.cpu().numpy()
    B[:steps, :steps] = r
    cols = r[:, 1:]
    if rank is not None:  # the dependent snapshot's coefficients close the last column
        last = (Q.T @ X[steps, :n].to(torch.float64)).cpu().numpy()
        cols = np.concatenate([cols, last[:, None]], 1)
    k = cols.shape[1]
    H[:steps, :k] = np.linalg.solve(r[:k, :k].T, cols.T).T
    return B, H, Q


def exact_solve(case, H, B, q, m, Q):
    beta, trunc = B[:m, :m], case["eig"] == "trunc"
    if trunc:
        U, sig, _ = np.linalg.svd(beta)
        r = int((sig > RANK_TOL * sig[0]).sum())
        U = U[:, :r]
        G = U.T @ H[:m, :m] @ U
    else:
        r, U, G = m, np.eye(m), H[:m, :m]
    lam, Z = np.linalg.eig(G)
    c = np.linalg.solve(Z, (B[0, 0] * U[0]).astype(complex))
    lab, ac = np.abs(lam), np.abs(c)
    pair = np.array([np.argmin(np.abs(lam - np.conj(x))) for x in lam])
    ac = np.maximum(ac, ac[pair])
    order = sorted(range(r), key=lambda i: (-round(ac[i] / ac.max(), 12), -round(lab[i], 10), -lam[i].imag))
    lam, c, Z = lam[order], c[order], Z[:, order]
    Y = U @ Z
    last = H[m, m - 1] if m < H.shape[0] else 0.0
    res = H[:m, :m] @ Y - U @ (G @ Z)
    ind = np.sqrt((np.abs(res) ** 2).sum(0) * (1 if trunc else 0) + (np.abs(last) * np.abs(Y[m - 1])) ** 2)
    out = {"r": None, "lam": lam, "amp": np.abs(c), "indicator": ind}
    if trunc:
        out["sigma"] = sig[:r]
    if case.get("vectors"):
        out["vec"] = Y[:, :case["vectors"]] * c[None, :case["vectors"]]
    if case.get("modes"):
        k = min(case["modes"], r)
        y = torch.from_numpy(Y[:, :k] * c[None, :k]).to(Q.device)
        out["modes_re"] = (y.real.T.contiguous() @ Q[:, :m].T)
        out["modes_im"] = (y.imag.T.contiguous() @ Q[:, :m].T)
    return out


def exact(case, seed):
    if case["kind"] == "streams":
        H, B = [], []
        for x, (n, N) in zip(stream_snapshots(case, seed), stream_sizes(case)):
            b, h, _ = projected(x, n)
            H.append(h.ravel())
            B.append(b.ravel())
        return {"q": None, "H": np.concatenate(H), "B": np.concatenate(B)}
    X = case_snapshots(case, seed)
    rank = 2 * case["waves"] if case["noise"] == 0.0 else None
    B, H, Q = projected(X, case["n"], rank)
    q = rank or case["N"]
    m = q if rank else q - 1
    out = {}
    if case["kind"] != "eig":
        out = {"q": None, "H": H, "B": B}
        if not case.get("modes"):
            out["V"] = Q.T
    if case.get("every"):
        out["indicators"] = None
    if case["eig"] != "none":
        out.update(exact_solve(case, H, B, q, m, Q))
    return out
