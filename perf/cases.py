"""Timed work of the library through its public entry points: block orthogonalization,
s-step GMRES, the matrix-powers kernel and the learned-preconditioner network.

Sizes are those of the benchmark and the tests (20000 x 60, 2^24 x 61 with s_hat = 30,
s = 10 / s_hat = 50 panels of 100 columns, Poisson 100^3, convection-diffusion 2048^2,
training instances of 512^2) and odd or smaller ones of the same kinds.  Inputs are
drawn on the GPU from the seed alone.  Solves run a fixed number of restart cycles
(the way the training data of the learned preconditioner are made), so that a pass is
the same work whatever the rounding.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_16717_gb300 as rbo


# ---- the cases -------------------------------------------------------------------------
def listed():
    return [
        # a small one-stage orthogonalization, bound by launches and reduction tails: the
        # CPU-checkable workload's shape
        dict(name="orth1-20000x60", kind="orth", n=20000, v0=0, s=5, nb=12, s_hat=0, d=244,
             kappa=1e4, prec="fp64"),
        # the precision sweep's matrix, one-stage: the largest orthogonalization
        dict(name="orth1-2^24x61", kind="orth", n=1 << 24, v0=1, s=5, nb=12, s_hat=0, d=244,
             kappa=1e4, prec="fp64"),
        # the same matrix through the two-stage scheme
        dict(name="orth2-2^24x61-30", kind="orth", n=1 << 24, v0=1, s=5, nb=12, s_hat=30, d=244,
             kappa=1e4, prec="fp64"),
        # the stress workload's panels (s = 10, s_hat = 50, m = 100) at an odd row count
        dict(name="orth2-1000003x101-50", kind="orth", n=1000003, v0=1, s=10, nb=10, s_hat=50,
             d=404, kappa=1e4, prec="fp64"),
        # mixed precision (float32 sketch and first projection) at an odd row count
        dict(name="orth1-mixed-4194301x61", kind="orth", n=4194301, v0=1, s=5, nb=12, s_hat=0,
             d=244, kappa=1e4, prec="mixed"),
        # a small solve, as in tests and prototyping: latency of every step of a cycle
        dict(name="gmres1-poisson20", kind="gmres", pde="poisson", N=20, s=5, s_hat=0, m=30,
             cycles=1, precond="jacobi", prec="fp64"),
        # the benchmark's solver configuration, one-stage
        dict(name="gmres1-poisson100", kind="gmres", pde="poisson", N=100, s=5, s_hat=0, m=60,
             cycles=2, precond="jacobi", prec="fp64"),
        # the benchmark's solver configuration, two-stage
        dict(name="gmres2-poisson100-20", kind="gmres", pde="poisson", N=100, s=5, s_hat=20, m=60,
             cycles=2, precond="jacobi", prec="fp64"),
        # evaluation solve of the learned preconditioner: values of M on A's pattern, s_hat = 30
        dict(name="gmres2-convdiff2048-M", kind="gmres", pde="convdiff", N=2048, s=5, s_hat=30,
             m=60, cycles=1, precond="M", prec="fp64"),
        # the matrix-powers kernel alone
        dict(name="mpk-poisson100", kind="mpk", pde="poisson", N=100, s=5),
        # inference of the learned preconditioner on an evaluation instance
        dict(name="gnn-infer-2048", kind="infer", pde="convdiff", N=2048),
        # loss and gradient on a training instance (6 residual columns + 4 probes)
        dict(name="gnn-grad-512", kind="grad", pde="convdiff", N=512, nr=10),
    ]


def _loguni(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["orth", "orth", "orth", "gmres", "gmres", "mpk", "infer", "grad"])
    if kind == "orth":
        s = rng.choice([2, 3, 4, 5, 5, 6, 8, 10])
        per = rng.choice([0, 2, 3, 4, 5, 6])  # panels per big panel (0: one-stage)
        while per and s * per > 60:
            per -= 1
        width = s * per if per else s
        nb = max(1, rng.randint(20, 100) // width) * (per if per else 1)
        v0 = rng.choice([0, 1])
        cols = v0 + nb * s
        n = _loguni(rng, 20000, (1 << 24) * 61 // max(cols, 61))
        prec = rng.choice(["fp64", "fp64", "fp64", "mixed"])
        return dict(kind="orth", n=n, v0=v0, s=s, nb=nb, s_hat=s * per, d=4 * (cols + 1),
                    kappa=10.0 ** rng.uniform(1, 4), prec=prec)
    if kind == "gmres":
        pde = rng.choice(["poisson", "poisson", "convdiff"])
        N = _loguni(rng, 32, 128) if pde == "poisson" else _loguni(rng, 128, 1500)
        s = rng.choice([2, 3, 4, 5, 5])
        per = rng.choice([0, 2, 3, 4])
        width = s * per if per else s
        m = width * max(1, rng.randint(30, 60) // width)
        return dict(kind="gmres", pde=pde, N=N, s=s, s_hat=s * per, m=m, cycles=1,
                    precond=rng.choice(["jacobi", "jacobi", "M"]), prec="fp64")
    if kind == "mpk":
        pde = rng.choice(["poisson", "convdiff"])
        N = _loguni(rng, 20, 160) if pde == "poisson" else _loguni(rng, 90, 2048)
        return dict(kind="mpk", pde=pde, N=N, s=rng.randint(2, 10))
    if kind == "infer":
        return dict(kind="infer", pde="convdiff", N=_loguni(rng, 64, 2048))
    return dict(kind="grad", pde="convdiff", N=_loguni(rng, 64, 700), nr=rng.randint(4, 10))


# ---- inputs ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _glued(case, seed):
    """The 'glued' matrix of the paper's experiments, transposed (row j = column j): an
    optional Gaussian start column, then blocks of s columns U diag(sigma) W^T, U Gaussian
    of unit column norm in expectation, sigma log-spaced from 1 to 1 / kappa, W orthogonal."""
    g = _gen(seed)
    n, s, nb, v0 = case["n"], case["s"], case["nb"], case["v0"]
    V = torch.empty((v0 + s * nb, n), device="cuda", dtype=torch.float64)
    if v0:
        V[0] = _randn(g, n)
    sig = torch.logspace(0.0, -math.log10(case["kappa"]), s, dtype=torch.float64, device="cuda")
    for j in range(nb):
        W, _ = torch.linalg.qr(_randn(g, s, s))
        U = _randn(g, s, n)
        torch.matmul(W * (sig / math.sqrt(n)), U, out=V[v0 + j * s:v0 + (j + 1) * s])
    return V


def _csr_from_stencil(cols, vals, ok):
    """CSR arrays from per-row candidates in ascending column order (n x k each)."""
    cnt = ok.sum(1)
    rowptr = torch.zeros(cols.shape[0] + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(cnt, 0)
    return rowptr, cols[ok], vals[ok]


def _poisson(N):
    """7-point Laplacian of an N^3 grid, Dirichlet boundaries."""
    i = torch.arange(N ** 3, device="cuda")
    x, y, z = i % N, (i // N) % N, i // (N * N)
    off = [(-N * N, z > 0), (-N, y > 0), (-1, x > 0), (0, x >= 0), (1, x < N - 1), (N, y < N - 1),
           (N * N, z < N - 1)]
    cols = torch.stack([i + o for o, _ in off], 1)
    ok = torch.stack([m for _, m in off], 1)
    vals = torch.full(cols.shape, -1.0, dtype=torch.float64, device="cuda")
    vals[:, 3] = 6.0
    return _csr_from_stencil(cols, vals, ok)


def _convdiff(N, seed):
    """2D convection-diffusion, 5-point upwind, N^2 cells: log-normal diffusivity (sigma 1,
    Gaussian correlation length 32 cells), constant wind of random angle, Peclet number
    uniform in [10, 1000]."""
    g = _gen(seed + 7919)
    f = _randn(g, N, N)
    q = torch.fft.fftfreq(N, device="cuda", dtype=torch.float64) * (2 * math.pi)
    filt = torch.exp(-0.5 * (32.0 / math.sqrt(2.0)) ** 2 * (q[:, None] ** 2 + q[None, :] ** 2))
    f = torch.fft.ifft2(torch.fft.fft2(f) * filt).real
    k = torch.exp((f - f.mean()) / f.std())
    u = torch.rand(2, generator=g, device="cuda", dtype=torch.float64).cpu()
    ang, pe = 2 * math.pi * float(u[0]), 10.0 + 990.0 * float(u[1])
    w = pe * float(k.mean())
    wx, wy = w * math.cos(ang), w * math.sin(ang)
    h = 1.0 / (N + 1)
    i = torch.arange(N * N, device="cuda")
    x, y = i % N, i // N
    kf = k.reshape(-1)

    def face(o, ok):
        j = torch.where(ok, i + o, i)
        return 2.0 * kf * kf[j] / (kf + kf[j])  # the cell's own value at the boundary

    sides = [(-N, y > 0, max(wy, 0.0)), (-1, x > 0, max(wx, 0.0)), (1, x < N - 1, max(-wx, 0.0)),
             (N, y < N - 1, max(-wy, 0.0))]
    c = [face(o, ok) / h ** 2 + conv / h for o, ok, conv in sides]
    vals = torch.stack([-c[0], -c[1], c[0] + c[1] + c[2] + c[3], -c[2], -c[3]], 1)
    cols = torch.stack([i - N, i - 1, i, i + 1, i + N], 1)
    ok = torch.stack([sides[0][1], sides[1][1], x >= 0, sides[2][1], sides[3][1]], 1)
    return _csr_from_stencil(cols, vals, ok)


def _matrix(case, seed):
    return _poisson(case["N"]) if case["pde"] == "poisson" else _convdiff(case["N"], seed)


def _rows(rowptr):
    n = rowptr.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device="cuda"), rowptr[1:] - rowptr[:-1])


def _device_csr(m):
    rowptr, col, val = (t.cpu().numpy() for t in m)
    return rbo.DeviceCSR(rowptr.size - 1, rowptr, col, val)


def _neumann(m):
    """Preconditioner values on A's pattern, D^-1 (2 I - A D^-1): the size and sign of what
    the trained network gives."""
    rowptr, col, val = m
    row = _rows(rowptr)
    d = torch.empty(rowptr.numel() - 1, dtype=torch.float64, device="cuda")
    d[row[row == col]] = val[row == col]
    return torch.where(row == col, 1.0 / d[row], -val / (d[row] * d[col]))


def _theta(seed):
    """Weights of the network: Gaussian matrices, small output weights and biases (the
    state of a network in training), in the library's parameter order."""
    r = np.random.default_rng(seed)
    out = []
    for kind, rows, cols in _SHAPES:
        sc = {"w": 0.5 * math.sqrt(2.0 / cols), "b": 0.05, "o": 0.1}[kind]
        out.append((r.standard_normal(rows * cols) * sc).astype(np.float32))
    return np.concatenate(out)


# parameter groups: encoder of nodes and edges, three layers (message, update), decoder
_SHAPES = ([("w", 32, 2), ("b", 32, 1), ("w", 32, 3), ("b", 32, 1)] +
           [("w", 32, 64), ("b", 32, 1), ("w", 32, 64), ("b", 32, 1)] * 3 + [("o", 1, 96), ("b", 1, 1)])


def _residuals(case, seed, n):
    R = rbo.colmajor(n, case["nr"])
    R.t().copy_(_randn(_gen(seed + 31), case["nr"], n))
    return R


def prepare(case, seed):
    kind = case["kind"]
    if kind == "orth":
        V0 = _glued(case, seed)
        V = rbo.colmajor(case["n"], V0.shape[0])
        return {"case": case, "V0": V0, "V": V, "sk": rbo.sketch_create(case["n"], case["d"], 8, 42)}
    m = _matrix(case, seed)
    A = _device_csr(m)
    st = {"case": case, "A": A}
    if kind in ("gmres", "mpk"):
        st["b"] = _randn(_gen(seed + 17), A.n)
        if case.get("precond") == "M":
            st["M"] = _neumann(m)
    if kind == "mpk":
        st["V"] = rbo.colmajor(A.n, case["s"])
    if kind in ("infer", "grad"):
        st["net"] = rbo.GNN(seed=0)
        st["net"].set_params(_theta(seed))
    if kind == "grad":
        st["R"] = _residuals(case, seed, A.n)
    return st


# ---- one pass ----------------------------------------------------------------------------
_PREC = {"fp64": rbo.PREC_FP64, "mixed": rbo.PREC_MIXED}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "orth":
        V = state["V"]
        V.t().copy_(state["V0"])  # the call overwrites V by Q: a pass starts from the data
        if case["s_hat"] > case["s"]:
            out = rbo.block_orth_two_stage(state["sk"], V, case["s"], case["s_hat"],
                                           v0=bool(case["v0"]), precision=_PREC[case["prec"]])
        else:
            out = rbo.block_orth_one_stage(state["sk"], V, case["s"], v0=bool(case["v0"]),
                                           precision=_PREC[case["prec"]])
        return [V.t(), out.R]
    if kind == "gmres":
        x, info = rbo.sstep_gmres(state["A"], state["b"], s=case["s"], s_hat=case["s_hat"],
                                  m=case["m"], tol=1e-10, max_restarts=case["cycles"],
                                  precond=0 if case["precond"] == "none" else 1,
                                  M=state.get("M"), precision=_PREC[case["prec"]])
        return [x, info["iterations"]]
    if kind == "mpk":
        return rbo.mpk_csr(state["A"], state["b"], case["s"], V=state["V"]).t()
    if kind == "infer":
        return state["net"].infer(state["A"])
    loss, grad = state["net"].loss_grad(state["A"], state["R"])
    return [loss, grad]


# ---- what a pass cannot do without -----------------------------------------------------
def work(case):
    if case["kind"] == "orth":
        n, c = case["n"], case["v0"] + case["s"] * case["nb"]
        # V read, Q written; two projections of every column against those before it
        return {"bytes": 16.0 * n * c, "flops": 4.0 * n * c * c}
    N = case["N"]
    n = N ** 3 if case["pde"] == "poisson" else N * N
    nnz = 7 * n - 6 * N * N if case["pde"] == "poisson" else 5 * n - 4 * N
    mat = 12.0 * nnz + 4.0 * n
    if case["kind"] == "gmres":
        its, m = case["cycles"] * case["m"], case["m"]
        # per iteration the operator applied and a column written; the basis read once per
        # cycle for x; two projections of every column
        op = mat + (8.0 * nnz if case["precond"] == "M" else 0.0)
        mv = 4.0 * nnz if case["precond"] == "M" else 2.0 * nnz
        return {"bytes": its * (op + 16.0 * n) + case["cycles"] * 8.0 * n * (m + 4),
                "flops": its * mv + case["cycles"] * 4.0 * n * m * m}
    if case["kind"] == "mpk":
        return {"bytes": mat + 8.0 * n * (case["s"] + 1), "flops": 2.0 * nnz * case["s"]}
    fw = nnz * 2.0 * (3 * 32 + 3 * 64 * 32 + 32) + n * 2.0 * (2 * 32 + 3 * 64 * 32 + 64)
    if case["kind"] == "infer":
        return {"bytes": mat + 8.0 * nnz, "flops": fw}
    return {"bytes": mat + 8.0 * n * case["nr"], "flops": 3.0 * fw + 8.0 * nnz * case["nr"]}


# ---- the same results in plain float64 torch ---------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "orth":
        return _exact_orth(_glued(case, seed))
    m = _matrix(case, seed)
    n = m[0].numel() - 1
    if kind == "mpk":
        A = torch.sparse_csr_tensor(*m, size=(n, n))
        v, out = _randn(_gen(seed + 17), n), []
        for _ in range(case["s"]):
            v = A @ v
            out.append(v)
        return torch.stack(out)
    if kind == "gmres":
        return [_exact_gmres(case, m, _randn(_gen(seed + 17), n)), case["cycles"] * case["m"]]
    theta = torch.from_numpy(_theta(seed)).cuda().to(torch.bfloat16).to(torch.float64)
    if kind == "infer":
        with torch.no_grad():
            return _exact_values(m, theta)
    theta.requires_grad_(True)
    M = _exact_values(m, theta)
    R = _randn(_gen(seed + 31), case["nr"], n).t()
    rowptr, col, val = m
    row = _rows(rowptr)

    def spmm(v, X):
        return torch.zeros_like(X).index_add(0, row, v[:, None] * X[col])

    E = R - spmm(val, spmm(M, R))
    loss = (E.square().sum(0) / R.square().sum(0)).mean()
    loss.backward()
    return [float(loss), theta.grad]


def _exact_orth(V):
    """QR of V (rows are columns here) by Cholesky QR three times: Q has orthonormal
    columns and R a positive diagonal, which makes both unique."""
    R = None
    for _ in range(3):
        L = torch.linalg.cholesky(V @ V.t())
        V = torch.linalg.solve_triangular(L, V, upper=False)
        R = L.t() if R is None else L.t() @ R
    return [V, R.cpu().numpy()]


def _exact_gmres(case, m, b):
    """Restarted GMRES with Arnoldi by twice-applied classical Gram-Schmidt."""
    rowptr, col, val = m
    n = b.numel()
    A = torch.sparse_csr_tensor(rowptr, col, val, size=(n, n))
    if case["precond"] == "M":
        Mm = torch.sparse_csr_tensor(rowptr, col, _neumann(m), size=(n, n))
    else:
        row = _rows(rowptr)
        d = torch.ones(n, dtype=torch.float64, device="cuda")
        d[row[row == col]] = val[row == col]
        Mm = None
    pre = (lambda v: Mm @ v) if Mm is not None else (lambda v: v / d)
    x, k = torch.zeros_like(b), case["m"]
    for _ in range(case["cycles"]):
        Q = torch.zeros((k + 1, n), dtype=torch.float64, device="cuda")
        H = torch.zeros((k + 1, k), dtype=torch.float64, device="cuda")
        r = b - A @ x
        beta = r.norm()
        Q[0] = r / beta
        for j in range(k):
            w = A @ pre(Q[j])
            for _ in range(2):
                h = Q[:j + 1] @ w
                w = w - h @ Q[:j + 1]
                H[:j + 1, j] += h
            H[j + 1, j] = w.norm()
            Q[j + 1] = w / H[j + 1, j]
        e = torch.zeros((k + 1, 1), dtype=torch.float64, device="cuda")
        e[0] = beta
        z = torch.linalg.lstsq(H, e).solution[:, 0]
        x = x + pre(z @ Q[:k])
    return x


def _exact_values(m, theta):
    """The network's values of M on A's pattern (width 32, three message-passing layers)."""
    rowptr, col, val = m
    n = rowptr.numel() - 1
    row = _rows(rowptr)
    p, o = [], 0
    for _, r, c in _SHAPES:
        p.append(theta[o:o + r * c].reshape(r, c))
        o += r * c
    dia = torch.empty(n, dtype=torch.float64, device="cuda")
    dia[row[row == col]] = val[row == col]
    tpos = torch.argsort(col * n + row)         # position of (j, i) for every (i, j)
    ah = val / dia[row]
    at = ah[tpos]
    offd = (row != col).to(torch.float64)
    zero = torch.zeros(n, dtype=torch.float64, device="cuda")
    f = torch.stack([zero.index_add(0, row, ah.abs() * offd), zero.index_add(0, row, at.abs() * offd)], 1)
    h = torch.relu(f @ p[0].t() + p[1][:, 0])
    e = torch.relu(torch.stack([ah, at, 1.0 - offd], 1) @ p[2].t() + p[3][:, 0])
    for l in range(3):
        wm, bm, wh, bh = p[4 + 4 * l:8 + 4 * l]
        msg = torch.relu(e @ wm[:, :32].t() + (h @ wm[:, 32:].t())[col] + bm[:, 0])
        agg = torch.zeros_like(h).index_add(0, row, msg)
        h = h + torch.relu(h @ wh[:, :32].t() + agg @ wh[:, 32:].t() + bh[:, 0])
        e = e + msg
    wo, bo = p[-2][0], p[-1][0, 0]
    out = e @ wo[:32] + (h @ wo[32:64])[row] + (h @ wo[64:])[col] + bo + (1.0 - offd)
    return out / dia[row]
