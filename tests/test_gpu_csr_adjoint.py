"""The CSR adjoint's fused products: gradients for column counts at the edges of the lane groups
(2, 4, 8, 16 lanes) and of the 16-column passes, rows shorter and longer than a batch of eight entries
and empty rows, against dense FP64 formulas on the returned X and Lambda (rounding only: rows of
at most 40 entries, sums over at most 33 columns, so 1e-12 of the largest entry)."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import to_device

pytestmark = pytest.mark.gpu


def _ragged(m, n, seed):
    rng = np.random.default_rng(seed)
    lens = rng.choice([0, 1, 3, 7, 8, 9, 17, 40], size=m)
    lens[:n] = np.maximum(lens[:n], 1)
    rp = np.zeros(m + 1, np.int64)
    np.cumsum(lens, out=rp[1:])
    ci = np.empty(rp[-1], np.int32)
    for i in range(m):
        c = rng.choice(n, size=lens[i], replace=False)
        if i < n and i not in c:
            c[0] = i
        ci[rp[i]:rp[i + 1]] = np.sort(c)
    return {"kind": "csr", "m": m, "n": n, "row_ptr": rp, "col_idx": ci, "vals": rng.standard_normal(rp[-1])}


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 16, 17, 33])
def test_csr_adjoint_products(lsq, k, dtype):
    mat = _ragged(3001, 50, 7)
    Mx, keep, seen = to_device(lsq, mat, dtype, with_f64=dtype == "f32")
    o = lsq.opts(seed=2, sample_factor=1.0, precond_dtype=1 if dtype == "f32" else 0)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    P = lsq.lsq_build_precond(Mx, idx, p, d, o)
    rng = np.random.default_rng(k)
    B = torch.from_numpy(rng.standard_normal((k, 3001))).cuda()
    X, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    G = torch.from_numpy(rng.standard_normal((k, 50))).cuda()
    gb, gv, lam, ai = lsq.lsq_pcg_adjoint(Mx, P, X, B, G, o)
    A = W.dense_from_csr(seen)
    Xh, Bh, L = X.cpu().numpy().reshape(k, -1), B.cpu().numpy(), lam.cpu().numpy()
    AL, R = L @ A.T, Bh - Xh @ A.T
    np.testing.assert_allclose(gb.cpu().numpy(), AL, rtol=0, atol=1e-12 * np.abs(AL).max())
    rows = np.repeat(np.arange(3001), np.diff(mat["row_ptr"]))
    ref = np.einsum("ce,ce->e", R[:, rows], L[:, mat["col_idx"]]) - np.einsum("ce,ce->e", AL[:, rows], Xh[:, mat["col_idx"]])
    np.testing.assert_allclose(gv.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
    assert np.linalg.norm(A.T @ (A @ L.T) - G.cpu().numpy().T) <= 1e-8 * np.linalg.norm(G.cpu().numpy())
