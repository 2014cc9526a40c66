"""Performance cases: what users of the solver have it do, through `paper_1806_02968_gb300.api`.

Six kinds of work, each over the range of sizes that the workloads, tests and benchmark of this
repository use:

* ``solve``  Alg. 2 end to end on a dense matrix (`api.solve`): sampling, preconditioner, PCG.
* ``pcg``    the solve alone on a handle that is kept, dense, one or several right-hand sides.
* ``setup``  sampling, the preconditioner and one application of it (a new matrix comes in).
* ``csr``    the solve alone on a kept handle, CSR (random rows or a weighted graph).
* ``grad``   the differentiable solve, forward and backward (`api.lsq_solve`).
* ``batch``  many small dense problems in one launch (`api.Batch`).

Inputs are drawn on the GPU from the seed: the same families as `workloads` (Gaussian, UDV,
semi-Gaussian, sparse random rows of very different norms, weighted graph incidence), with
b = A x* + noise.  Tolerances are the benchmark's 1e-10 where the matrix is well conditioned and
1e-13 where it is not, so that the solution is determined to far below the tolerance of a
comparison.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_02968_gb300 import api

F64, F32 = torch.float64, torch.float32
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f32x2": 8}


def listed():
    return [
        # The smallest whole call: the Gaussian example of the smoke run (0.5 M values, in L2);
        # launches, synchronisations and grid barriers.
        dict(name="solve_gauss_4096x128", kind="solve", matrix="gauss", m=4096, n=128, dtype="f64",
             k=1, sweeps=1, kappa=1.0, tol=1e-10),
        # A whole call at the largest row of the Gaussian table of Sec. 5.1 with the paper's
        # five sweeps: sampling and building the operator weigh as much as the iteration.
        dict(name="solve_gauss_40000x400_t5", kind="solve", matrix="gauss", m=40000, n=400, dtype="f64",
             k=1, sweeps=5, kappa=1.0, tol=1e-10),
        # Sec. 5.4's UDV size in FP64, moderately conditioned: a new right-hand side for a
        # matrix whose handle is kept.
        dict(name="pcg_udv_90000x300_f64", kind="pcg", matrix="udv", m=90000, n=300, dtype="f64",
             k=1, sweeps=1, kappa=100.0, tol=1e-13),
        # The benchmark's matrix and value type (double-float pairs, FP64 copy for the true
        # residual) at a condition number that fits a pass: the HBM-bound iteration.
        dict(name="pcg_udv_262144x512_f32x2", kind="pcg", matrix="udv", m=262144, n=512, dtype="f32x2",
             k=1, sweeps=1, kappa=100.0, tol=1e-13),
        # The FP32 precision form on a ragged matrix with a padded leading dimension and a
        # block of eight right-hand sides.
        dict(name="pcg_gauss_60001x201_f32_k8", kind="pcg", matrix="gauss", m=60001, n=201, dtype="f32",
             k=8, sweeps=1, kappa=1.0, tol=1e-10),
        # BF16 values on a well-conditioned matrix (wide rows, half the bytes of FP32).
        dict(name="pcg_gauss_100000x1000_bf16", kind="pcg", matrix="gauss", m=100000, n=1000, dtype="bf16",
             k=1, sweeps=1, kappa=1.0, tol=1e-10),
        # Setup for the benchmark's matrix: three passes over A, 12777 draws, A_s^T A_s and the
        # operator.
        dict(name="setup_udv_262144x512_f64", kind="setup", matrix="udv", m=262144, n=512, dtype="f64",
             k=1, sweeps=1, kappa=100.0, tol=1e-13),
        # Setup for the sparse benchmark matrix: draws from four million rows, the SpGEMM, the
        # level schedules and the transposed pattern.
        dict(name="setup_sprand_4Mx40k_f32", kind="setup", matrix="sprand", m=4000000, n=40000, dtype="f32",
             k=1, sweeps=1, kappa=1.0, tol=1e-10),
        # The sparse benchmark solve: one right-hand side, FP32 values and operator, FP64
        # restarts.
        dict(name="csr_sprand_4Mx40k_f32", kind="csr", matrix="sprand", m=4000000, n=40000, dtype="f32",
             k=1, sweeps=1, kappa=1.0, tol=1e-10),
        # The graph workload: 32 right-hand sides of a weighted incidence matrix in one
        # persistent launch.
        dict(name="csr_graph_262144_f64_k32", kind="csr", matrix="graph", m=8 * 262144, n=262143, dtype="f64",
             k=32, sweeps=1, kappa=1.0, tol=1e-12),
        # Training through the sparse solve: 16 right-hand sides, forward and backward, gradients
        # of the values and of the right-hand sides.
        dict(name="grad_sprand_1Mx10k_f32_k16", kind="grad", matrix="sprand", m=1000000, n=10000, dtype="f32",
             k=16, sweeps=1, kappa=1.0, tol=1e-10),
        # 64 uneven small problems with 16 right-hand sides each in one launch.
        dict(name="batch_64x16rhs", kind="batch", matrix="gauss", count=64, k=16, m_lo=1024, m_hi=16384,
             n_lo=32, n_hi=256, dtype="f32", sweeps=1, kappa=1.0, tol=1e-10),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "pcg", "pcg", "setup", "setup", "csr", "csr", "grad", "grad", "batch"])
    c = dict(kind=kind, k=1, sweeps=1, kappa=1.0, tol=1e-10)
    if kind == "batch":
        c.update(matrix="gauss", dtype="f32", count=rng.randint(8, 64), k=rng.randint(1, 16),
                 m_lo=1024, m_hi=log_int(2048, 16384), n_lo=32, n_hi=log_int(48, 256))
        return c
    sparse = kind == "csr" or (kind in ("setup", "grad") and rng.random() < 0.5)
    if not sparse:
        n = log_int(40, 1000)
        m = log_int(max(1000, 6 * n), max(2000, min(262144, 134000000 // n)))
        c["matrix"] = rng.choice(["gauss", "udv", "semi"])
        c["dtype"] = "f64"
        if kind == "pcg":
            c["dtype"] = rng.choice(["f64", "f32x2", "f32", "bf16"])
            c["k"] = rng.choice([1, 1, 2, 5, 8])
        elif kind == "grad":
            c["dtype"] = rng.choice(["f64", "f32"])
            c["k"] = rng.randint(1, 8)
            n = max(40, n // 4 * 4)      # the differentiable solve takes unpadded rows
            m = min(m, 20000000 // n)
        elif kind == "setup":
            c["dtype"] = rng.choice(["f64", "f32"])
            c["sweeps"] = rng.choice([1, 2])
        else:
            n = min(n, 512)
            c["sweeps"] = rng.choice([1, 2, 5])
        if c["dtype"] in ("f32", "bf16") and kind in ("pcg", "grad"):
            c["matrix"] = "gauss"
        if c["matrix"] == "udv":
            c["kappa"], c["tol"] = float(round(10.0 ** rng.uniform(0.5, 2.0), 2)), 1e-13
        c.update(m=m, n=n)
        return c
    c["matrix"] = rng.choice(["sprand", "sprand", "graph"])
    c["dtype"] = rng.choice(["f64", "f32"])
    if c["matrix"] == "graph":
        n = log_int(2000, 262143)
        c.update(m=8 * (n + 1) - rng.randint(0, 99), n=n, dtype="f64", tol=1e-12)
        if kind == "csr":
            c["k"] = rng.choice([2, 8, 16, 32])
    else:
        n = log_int(300, 10000 if kind == "grad" else 40000)
        c.update(m=min(log_int(50 * n, 200 * n), 4000000 if kind != "grad" else 1000000), n=n)
        if kind == "csr":
            c["k"] = 1 if n > 4000 else rng.choice([1, 4, 16])
    if kind == "grad":
        c["k"] = rng.choice([2, 8, 16]) if c["n"] <= 10000 else 2
    return c


# -- inputs -----------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 62) + 17)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=F64)


def _dense(g, case, m, n):
    """Gaussian; UDV with sigma log-spaced from 1 to 1/kappa; semi-Gaussian [B 0; 0 I]."""
    G = _randn(g, m, n)
    if case["matrix"] == "semi":
        h = n // 2
        G[:, h:] = 0.0
        G[m - (n - h):, :] = 0.0
        G[m - (n - h):, h:] = torch.eye(n - h, dtype=F64, device="cuda")
    elif case["matrix"] == "udv":
        V = np.linalg.qr(_randn(g, n, n).cpu().numpy())[0]
        R = np.linalg.cholesky((G.T @ G).cpu().numpy()).T
        sigma = np.logspace(0.0, -math.log10(case["kappa"]), n)
        G = G @ torch.from_numpy(np.linalg.solve(R, sigma[:, None] * V.T)).cuda()
    return G


def _stored(G, dtype):
    """The matrix as a user stores it (rows padded to 16 bytes) and the FP64 values it stands for."""
    m, n = G.shape
    per = 16 // VALUE_BYTES[dtype]
    ld = max((n + per - 1) // per * per, (n + 1) // 2 * 2)
    if dtype == "f64":
        T = torch.zeros(m, ld, dtype=F64, device="cuda")
        T[:, :n] = G
        return api.Matrix(T[:, :n]), T[:, :n]
    F = torch.zeros(m, ld, dtype=F64, device="cuda")
    if dtype == "f32x2":
        F[:, :n] = G
        return api.Matrix(api.lsq_split_f64(F)[:, :2 * n], f32x2=True, vals_f64=F), F[:, :n]
    T = torch.zeros(m, ld, dtype=F32 if dtype == "f32" else torch.bfloat16, device="cuda")
    T[:, :n] = G.to(T.dtype)
    F[:, :n] = T[:, :n].double()
    return api.Matrix(T[:, :n], vals_f64=F), F[:, :n]


def _csr(g, case):
    """(row_ptr, col_idx, vals, rows): random rows of 8 entries and very different norms with
    every column present, or the incidence rows of a connected weighted graph, one vertex
    grounded.  The number of entries goes with the case, not with the seed."""
    m, n = case["m"], case["n"]

    def randint(hi, *shape):
        return torch.randint(0, hi, shape, generator=g, device="cuda")

    def uniform(size, lo, hi):
        return lo + (hi - lo) * torch.rand(size, generator=g, device="cuda", dtype=F64)

    if case["matrix"] == "graph":
        # vertex 0 (grounded, its column left out) has 16 edges; the others are joined by a path
        src, dst = 1 + randint(n, m), randint(n - 1, m)
        dst = 1 + (src + dst) % n
        src[:16] = 0
        path = 1 + torch.randperm(n, generator=g, device="cuda")
        src, dst = torch.cat([src, path[:-1]]), torch.cat([dst, path[1:]])
        w = torch.sqrt(10.0 ** uniform(src.numel(), -3.0, 3.0))
        m = src.numel()
        rows = torch.arange(m, device="cuda")
        rows, cols, vals = torch.cat([rows, rows]), torch.cat([src, dst]), torch.cat([w, -w])
        keep = cols > 0
        key, at = torch.sort(rows[keep] * n + cols[keep] - 1)
        vals = vals[keep][at]
    else:
        cols = torch.sort(randint(n, m, 8), dim=1).values
        while True:
            bad = (cols[:, 1:] == cols[:, :-1]).any(1).nonzero()[:, 0]
            if bad.numel() == 0:
                break
            cols[bad] = torch.sort(randint(n, bad.numel(), 8), dim=1).values
        # every column once more, eight to a row, in rows of their own
        every = torch.randperm(n, generator=g, device="cuda")
        every = torch.cat([every, every[:-n % 8]]).reshape(-1, 8)
        cols[torch.randperm(m, generator=g, device="cuda")[:every.shape[0]]] = torch.sort(every, dim=1).values
        key = (torch.arange(m, device="cuda")[:, None] * n + cols).reshape(-1)
        scale = 10.0 ** uniform(m, -2.0, 2.0)
        vals = _randn(g, key.numel()) * scale[key // n]
    rows = key // n
    row_ptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return row_ptr, (key % n).to(torch.int32), vals, rows


def _csr_times(row_ptr, col, vals, X):
    """A X^T for X (k, n) in FP64, entry by entry of every row (a fixed order): (k, m)."""
    out = torch.zeros(X.shape[0], row_ptr.numel() - 1, dtype=F64, device="cuda")
    start, length = row_ptr[:-1], row_ptr[1:] - row_ptr[:-1]
    for j in range(int(length.max())):
        has = (length > j).nonzero()[:, 0]
        e = start[has] + j
        out[:, has] += vals[e].double() * X[:, col[e].long()]
    return out


def _opts(case, seed, small_operator):
    refine = case["dtype"] in ("f32", "bf16") and case["kind"] != "setup"
    kw = dict(seed=int(seed) % (1 << 31) + 7, tol=case["tol"], sweeps=case["sweeps"], maxit=100000, max_outer=50,
              precond_dtype=1 if small_operator else 0)
    if refine and case["matrix"] != "sprand":
        kw["inner_tol"] = 1e-4
    if case["kind"] == "csr" and case["matrix"] == "graph":
        kw["device_loop"] = 1
    return api.opts(**kw)


def _handle(Mx, o):
    idx, p, d = api.lsq_sample_rows(Mx, o)
    return api.lsq_build_precond(Mx, idx, p, d, o)


def _batch_sizes(case, seed):
    rng = np.random.default_rng(int(seed))
    return [(int(round(math.exp(rng.uniform(math.log(case["m_lo"]), math.log(case["m_hi"]))))),
             int(round(math.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))))
            for _ in range(case["count"])]


def _inputs(case, seed):
    """The user's data: matrix, its FP64 values, right-hand sides, and for ``grad`` the
    incoming gradient."""
    g = _gen(seed)
    k = case["k"]
    s = {}
    if case["kind"] == "batch":
        s["problems"] = []
        # the sizes go with the case (every seed has the same work), the values with the seed
        for m, n in _batch_sizes(case, case["count"]):
            T = torch.zeros(m, (n + 3) // 4 * 4, dtype=F32, device="cuda")
            T[:, :n] = _randn(g, m, n).float()
            A = T[:, :n].double()
            B = (A @ _randn(g, n, k)).T + 1e-3 * _randn(g, k, m)
            s["problems"].append((T, n, A, B.contiguous()))
        return s
    if case["matrix"] in ("sprand", "graph"):
        rp, ci, v, rows = _csr(g, case)
        vals = v.float() if case["dtype"] == "f32" else v
        F = vals.double() if case["dtype"] == "f32" else None
        s["A"] = api.Matrix(row_ptr=rp, col_idx=ci, vals=vals, n=case["n"], vals_f64=F)
        s["exact"] = (rp, ci, vals.double(), rows)
        m = rp.numel() - 1
        if case["kind"] != "setup":
            s["B"] = _csr_times(rp, ci, vals, _randn(g, k, case["n"])) + 1e-3 * _randn(g, k, m)
    else:
        m = case["m"]
        s["A"], s["exact"] = _stored(_dense(g, case, m, case["n"]), case["dtype"])
        if case["kind"] != "setup":
            s["B"] = ((s["exact"] @ _randn(g, case["n"], k)).T + 1e-3 * _randn(g, k, m)).contiguous()
    if case["kind"] == "grad":
        s["G"] = _randn(g, k, case["n"])
    if case["kind"] == "setup":
        s["R"] = _randn(g, case["n"])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s.pop("exact", None)
    s["kind"] = case["kind"]
    if case["kind"] == "batch":
        o = api.opts(tol=case["tol"], maxit=100000, max_outer=30, inner_tol=1e-4)
        problems = []
        for i, (T, n, A, B) in enumerate(s.pop("problems")):
            P = _handle(api.Matrix(T[:, :n]), api.opts(seed=200 + i, precond_dtype=1))
            problems.append((T, n, P, B))
        s["batch"] = api.Batch(problems, o)
        return s
    A = s["A"]
    s["o"] = o = _opts(case, seed, case["dtype"] in ("f32", "bf16"))
    if case["kind"] in ("pcg", "csr", "grad"):
        s["P"] = _handle(A, o)
    if case["kind"] == "solve":
        s["B"] = s["B"][0]
    if case["kind"] == "grad":
        s["vals"] = A.vals.requires_grad_(True)
        s["B"].requires_grad_(True)
    return s


def run(s):
    kind = s["kind"]
    if kind == "solve":
        x, _, more = api.solve(s["A"], s["B"], s["o"])
        return {"x": x, "idx": more["idx"], "p": more["p"], "d": more["colscale"]}
    if kind in ("pcg", "csr"):
        X, _ = api.lsq_pcg_solve(s["A"], s["P"], s["B"], s["o"])
        return {"x": X}
    if kind == "setup":
        idx, p, d = api.lsq_sample_rows(s["A"], s["o"])
        P = api.lsq_build_precond(s["A"], idx, p, d, s["o"])
        return {"idx": idx, "p": p, "d": d, "z": P.apply(s["R"])}
    if kind == "grad":
        X = api.lsq_solve(s["A"], s["B"], s["P"], s["o"])
        gv, gb = torch.autograd.grad(X, [s["vals"], s["B"]], s["G"])
        return {"x": X.detach(), "grad_vals": gv, "grad_b": gb}
    s["batch"].solve()
    return {"x": list(s["batch"].X)}


# -- what a pass cannot do without ---------------------------------------------------------------

def _iterations(case):
    """About how many PCG iterations the method takes (measured; well-conditioned matrices and
    moderately conditioned ones)."""
    if case["matrix"] == "graph":
        return 90
    if case["matrix"] == "udv":
        return int(16 + 5.3 * case["kappa"])
    return 16 if case["tol"] >= 1e-10 else 20


def work(case):
    k, its = case["k"], _iterations(case)
    es = VALUE_BYTES[case["dtype"]]
    if case["kind"] == "batch":
        b = f = 0.0
        for m, n in _batch_sizes(case, case["count"]):
            b += 4.0 * m * n + 8.0 * k * (m + n) + 4.0 * n * n
            f += its * k * (4.0 * m * n + 2.0 * n * n)
        return {"bytes": b, "flops": f}
    m, n = case["m"], case["n"]
    s = math.ceil(4 * n * math.log(n))
    if case["matrix"] in ("sprand", "graph"):
        if case["matrix"] == "graph":
            m, per = m + n, 2
        else:
            per = 8
        nnz = float(m * per)
        nnz_m = min(n + min(s, m) * per * (per - 1.0), float(n) * n)
        sampling = nnz * (es + 4) + 16.0 * m + 4.0 * s
        build = nnz * (4 + 4) + s * per * (es + 4.0) + nnz_m * 12
        iteration = nnz * (es + 4) + nnz_m * (es + 4) + 80.0 * n * k
        flops = k * (4.0 * nnz + 2.0 * nnz_m)
        small = 2.0 * s * per * per
    else:
        nnz = float(m) * n
        sampling = nnz * es + 16.0 * m
        build = float(s) * n * es + 8.0 * n * n
        iteration = nnz * es + es * n * n
        flops = k * (4.0 * nnz + 2.0 * n * n)
        small = float(s) * n * n + 2.0 * case["sweeps"] * 2.0 * n ** 3
    # the matrix is larger than the L2 cache in some cases only; there every iteration has to
    # read it again
    again = its if nnz * es > 1.2e8 else 1
    solve = (iteration * again + 8.0 * k * (m + n), flops * its)
    if case["kind"] == "setup":
        return {"bytes": sampling + build, "flops": 3.0 * nnz + small}
    if case["kind"] == "solve":
        return {"bytes": sampling + build + solve[0], "flops": 3.0 * nnz + small + solve[1]}
    if case["kind"] == "grad":
        return {"bytes": 2 * solve[0] + nnz * (es + 8) + 24.0 * m * k, "flops": 2 * solve[1] + 8.0 * nnz * k}
    return {"bytes": solve[0], "flops": solve[1]}


# -- the same in 64 bits ------------------------------------------------------------------------

def _chol_solver(A):
    L = np.linalg.cholesky((A.T @ A).cpu().numpy())
    Li = np.linalg.inv(L)
    inv = torch.from_numpy(Li.T @ Li).cuda()

    def normal(H):               # (A^T A)^-1 H, refined; H is (n, k)
        Y = inv @ H
        for _ in range(3):
            Y = Y + inv @ (H - A.T @ (A @ Y))
        return Y

    def least_squares(B):        # B is (m, k)
        Y = inv @ (A.T @ B)
        for _ in range(3):
            Y = Y + inv @ (A.T @ (B - A @ Y))
        return Y
    return normal, least_squares


def _csr_exact(exact, n):
    """The same two solvers for CSR, by conjugate gradients with diagonal scaling, restarted
    from the true residual until it stops falling."""
    rp, ci, v, rows = exact
    col = ci.long()
    d = torch.sqrt(torch.zeros(n, dtype=F64, device="cuda").index_add_(0, col, v * v))

    def times(X):                # (n, k) -> (m, k)
        return _csr_times(rp, ci, v, X.T.contiguous()).T

    def back(Q):                 # (m, k) -> (n, k)
        return torch.zeros(n, Q.shape[1], dtype=F64, device="cuda").index_add_(0, col, v[:, None] * Q[rows])

    def cg(H):
        g = H / d[:, None]
        y, p, rho = torch.zeros_like(g), g.clone(), (g * g).sum(0)
        start = rho.clone()
        for it in range(3000):
            w = back(times(p / d[:, None])) / d[:, None]
            alpha = torch.where(rho > 0, rho / (p * w).sum(0).clamp_min(1e-300), rho)
            y += alpha * p
            g -= alpha * w
            new = (g * g).sum(0)
            if it % 10 == 9 and bool((new <= 1e-18 * start).all()):
                break
            p = g + torch.where(rho > 0, new / rho.clamp_min(1e-300), rho) * p
            rho = new
        return y / d[:, None]

    def normal(H):
        Y = cg(H)
        for _ in range(2):
            Y = Y + cg(H - back(times(Y)))
        return Y

    def least_squares(B):
        Y = cg(back(B))
        for _ in range(2):
            Y = Y + cg(back(B - times(Y)))
        return Y
    return normal, least_squares, times, d


def exact(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    if kind == "batch":
        return {"x": [_chol_solver(A)[1](B.T).T.contiguous() for _, _, A, B in s["problems"]]}
    e = s["exact"]
    sparse = case["matrix"] in ("sprand", "graph")
    if kind == "setup":          # the draws have no outside reference; the column norms have
        if sparse:
            rp, ci, v, rows = e
            d2 = torch.zeros(case["n"], dtype=F64, device="cuda").index_add_(0, ci.long(), v * v)
        else:
            d2 = (e * e).sum(0)
        return {"idx": None, "p": None, "d": torch.sqrt(d2), "z": None}
    if sparse:
        normal, least_squares, times, _ = _csr_exact(e, case["n"])
    else:
        normal, least_squares = _chol_solver(e)
        times = e.matmul
    X = least_squares(s["B"].T)
    if kind == "solve":
        return {"x": X[:, 0].contiguous(), "idx": None, "p": None, "d": torch.sqrt((e * e).sum(0))}
    if kind != "grad":
        return {"x": X.T.contiguous()}
    Lam = normal(s["G"].T)
    AL, R = times(Lam), s["B"].T - times(X)
    if sparse:
        rp, ci, v, rows = e
        gv = torch.zeros_like(v)
        for c in range(case["k"]):
            gv += R[rows, c] * Lam[ci.long(), c] - AL[rows, c] * X[ci.long(), c]
    else:
        gv = R @ Lam.T - AL @ X.T
    return {"x": X.T.contiguous(), "grad_vals": gv, "grad_b": AL.T.contiguous()}
