"""Gauss-Seidel sweeps by blocks of rows (deep level schedules, the form chosen by shape): sizes at
the edges of the 64- and 128-row blocks, one and several sweeps, FP64 and FP32 M, and blocks of
right-hand sides that fill and do not fill a group of columns.

Tolerances: those of the row forms on the same quantities.  FP64 M against the oracle's literal
Alg. 3 at 1e-11; FP32 M (double-float sums, ~48 bits) against Alg. 3 in FP64 on the same matrix
at 1e-10."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import assert_solution, rel, to_device
from test_gpu_sparse import _sgs_reference

pytestmark = pytest.mark.gpu


def _handle(lsq, mat, dtype="f64", **kw):
    Mx, keep, seen = to_device(lsq, mat, dtype, with_f64=dtype == "f32")
    o = lsq.opts(seed=11, **kw)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    return Mx, keep, seen, o, lsq.lsq_build_precond(Mx, idx, p, d, o)


def _levels(rp, ci, n):
    lev = np.zeros(n, np.int64)
    for j in range(n):
        dep = ci[rp[j]:rp[j + 1]]
        dep = dep[dep < j]
        lev[j] = 1 + lev[dep].max() if dep.size else 0
    return int(lev.max()) + 1


@pytest.mark.parametrize("sweeps", [1, 2])
@pytest.mark.parametrize("n", [8, 63, 64, 65, 127, 128, 129, 191, 257, 1000])
def test_blocked_sweeps_match_alg3(lsq, orc, n, sweeps):
    mat = W.sparse_random(60 * n, n, 8, n)
    Mx, keep, seen, o, P = _handle(lsq, mat, sweeps=sweeps)
    rp, ci, va = (t.cpu().numpy() for t in P.M_csr())
    smp = orc.Sample(seen, seed=11)
    Mo = orc.SampledM(smp)
    assert np.array_equal(rp, Mo.row_ptr) and np.array_equal(ci, Mo.col)
    assert _levels(rp, ci, n) >= (n + 127) // 128           # the shape that takes this form
    R = np.random.default_rng(n).standard_normal((3, n))
    E = P.apply(torch.from_numpy(R).cuda()).cpu().numpy()
    for c in range(3):
        assert rel(E[c], orc.sgs_apply(Mo, R[c], sweeps)) <= 1e-11


@pytest.mark.parametrize("sweeps", [1, 3])
@pytest.mark.parametrize("n", [65, 128, 300, 1100])
def test_blocked_sweeps_fp32_m(lsq, orc, n, sweeps):
    import scipy.sparse as sps
    mat = W.sparse_random(60 * n, n, 8, n + 1)
    Mx, keep, seen, o, P = _handle(lsq, mat, sweeps=sweeps, precond_dtype=1)
    rp, ci, va = (t.cpu().numpy() for t in P.M_csr())
    rows = np.repeat(np.arange(n), np.diff(rp))
    M32 = sps.csr_matrix((np.where(rows == ci, va, va.astype(np.float32).astype(np.float64)), ci, rp), shape=(n, n))
    assert np.array_equal(M32.toarray(), M32.toarray().T)    # M is symmetric to the bit
    R = np.random.default_rng(n).standard_normal((2, n))
    E = P.apply(torch.from_numpy(R).cuda()).cpu().numpy()
    for c in range(2):
        assert rel(E[c], _sgs_reference(M32, R[c], sweeps)) <= 1e-10


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 17, 33])
def test_blocked_block_solve_matches_single_columns(lsq, orc, dtype, k):
    """Every column of a block of right-hand sides against the same column solved alone (the
    sweeps of both run by blocks of rows), and the first against the oracle."""
    mat = W.sparse_random(12000, 200, 8, 3)
    Mx, keep, seen, o, P = _handle(lsq, mat, dtype, precond_dtype=1 if dtype == "f32" else 0)
    xs, b = W.rhs_for(seen, k, 1e-3, 7)
    B = torch.from_numpy(b).cuda()
    X, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    X = X.cpu().numpy()
    smp = orc.Sample(seen, seed=11)
    kappa = np.linalg.cond(W.dense_from_csr(seen) / smp.d)
    for c in sorted({0, 1, k // 2, k - 1}):
        x1, i1 = lsq.lsq_pcg_solve(Mx, P, B[c], o)
        assert info.converged[c] == 1 and abs(int(info.iters[c]) - int(i1.iters[0])) <= 2
        assert_solution(X[c], x1.cpu().numpy(), kappa, f"column {c}")
    y, oi = orc.pcg(smp.mat, smp.d, orc.SampledM(smp), b=b[0], tol=o.tol, maxit=o.maxit, max_outer=o.max_outer)
    assert_solution(X[0], y / smp.d, kappa, "column 0 against the oracle")
