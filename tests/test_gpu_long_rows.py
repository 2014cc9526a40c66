"""CSR matrices of mostly short rows with a few long ones, which a whole CTA takes together: lengths at
the edge of what counts as long (1024 entries), several long rows in one warp, the last row long, and
whole warps of long rows."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import to_device

pytestmark = pytest.mark.gpu


def _matrix(mean, seed, many=False):
    """4000 rows, most of 1 to 2 `mean` entries; the long ones small, so that few of them are drawn."""
    rng = np.random.default_rng(seed)
    m, n = 4000, 1500
    lens = rng.integers(1, 2 * mean + 1, m)
    long = np.array([1, 2, 3, 500, 501, 1500, 1501, 2600, 2601, m - 1])
    lens[long] = [1023, 1024, 1025, 1500, 65, 1026, 1027, 1500, 257, 1500]
    if many:
        lens[700:1000] = 1025
        long = np.concatenate([long, np.arange(700, 1000)])
    rp = np.concatenate([[0], np.cumsum(lens)])
    ci = np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for k in lens])
    base = np.arange(n)                                # every column in a row of its own
    rp = np.concatenate([rp, rp[-1] + 1 + base])
    ci = np.concatenate([ci, base]).astype(np.int32)
    va = rng.standard_normal(rp[-1])
    for i in long:
        va[rp[i]:rp[i + 1]] *= 1e-6 if many else 1e-3
    return {"kind": "csr", "m": m + n, "n": n, "row_ptr": rp.astype(np.int64), "col_idx": ci, "vals": va}


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("mean", [1, 2, 5])
def test_sampling_with_long_rows(lsq, orc, mean, dtype):
    mat = _matrix(mean, mean)
    Mx, keep, seen = to_device(lsq, mat, dtype)
    idx, p, d = lsq.lsq_sample_rows(Mx, lsq.opts(seed=3))
    smp = orc.Sample(seen, seed=3)
    assert np.array_equal(idx.cpu().numpy(), smp.idx) and np.array_equal(d.cpu().numpy(), smp.d)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k,many", [(1, False), (3, False), (8, False), (17, False), (2, True)])
def test_solve_and_adjoint_with_long_rows(lsq, k, many, dtype):
    """Products and gradients against FP64 formulas on the returned X and Lambda: 1500 terms a sum, so
    1e-12 of the largest entry; the solution against the normal equations (the transposed pattern)."""
    mat = _matrix(2, 9, many)
    Mx, keep, seen = to_device(lsq, mat, dtype, with_f64=dtype == "f32")
    o = lsq.opts(seed=2, sample_factor=0.5)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    P = lsq.lsq_build_precond(Mx, idx, p, d, o)
    rng = np.random.default_rng(k)
    B = torch.from_numpy(rng.standard_normal((k, Mx.m))).cuda()
    G = torch.from_numpy(rng.standard_normal((k, Mx.n))).cuda()
    X, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    assert all(info.converged == 1)
    gb, gv, lam, ai = lsq.lsq_pcg_adjoint(Mx, P, X, B, G, o)
    A, Bh = W.dense_from_csr(seen), B.cpu().numpy()
    Xh, L = X.cpu().numpy(), lam.cpu().numpy()
    AL, R = L @ A.T, Bh - Xh @ A.T
    assert np.linalg.norm(R @ A) <= 1e-8 * np.linalg.norm(Bh @ A)
    np.testing.assert_allclose(gb.cpu().numpy(), AL, rtol=0, atol=1e-12 * np.abs(AL).max())
    rows = np.repeat(np.arange(Mx.m), np.diff(mat["row_ptr"]))
    ci = mat["col_idx"]
    ref = np.einsum("ce,ce->e", R[:, rows], L[:, ci]) - np.einsum("ce,ce->e", AL[:, rows], Xh[:, ci])
    np.testing.assert_allclose(gv.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
