"""Several right-hand sides of a dense matrix in one launch (groups of CTAs side by side): every
column as it comes out when it is solved alone, for counts that fill one round, need several and
leave groups idle, few rows, and the adjoint's normal form.

Two solves that meet the tolerance differ by at most the solution bar of the parity tests."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import assert_solution, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("m,n,k", [(40, 3, 5), (300, 20, 16), (3001, 70, 2), (3001, 70, 17), (5000, 130, 33)])
def test_dense_columns_match_single_solves(lsq, orc, m, n, k, dtype):
    mat = W.gaussian_dense(m, n, m + k)
    Mx, keep, seen = to_device(lsq, mat, dtype, with_f64=dtype == "f32", ld_pad=(-n) % 4)
    o = lsq.opts(seed=5, max_outer=30, inner_tol=1e-4 if dtype == "f32" else 0.0)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    P = lsq.lsq_build_precond(Mx, idx, p, d, o)
    xs, b = W.rhs_for(seen, k, 1e-3, 9)
    b[k // 2] = 0.0                                  # a zero column among the others
    B = torch.from_numpy(b).cuda()
    n0 = lsq.launches()
    X, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    assert lsq.launches() - n0 == 1
    kappa = np.linalg.cond(seen["A"] / d.cpu().numpy())
    assert np.all(X[k // 2].cpu().numpy() == 0.0) and info.iters[k // 2] == 0 and all(info.converged == 1)
    for c in sorted({0, 1, k - 1} - {k // 2}):
        x1, i1 = lsq.lsq_pcg_solve(Mx, P, B[c], o)
        assert abs(int(info.iters[c]) - int(i1.iters[0])) <= 2
        assert_solution(X[c].cpu().numpy(), x1.cpu().numpy(), kappa, f"column {c}")
        assert_solution(X[c].cpu().numpy(), np.linalg.lstsq(seen["A"], b[c], rcond=None)[0], kappa, f"column {c}")
    if dtype == "f64":
        G = torch.from_numpy(np.random.default_rng(1).standard_normal((k, n))).cuda()
        gb, gv, lam, ai = lsq.lsq_pcg_adjoint(Mx, P, X, B, G, o)
        ref = np.linalg.solve(seen["A"].T @ seen["A"], G.cpu().numpy().T).T
        for c in sorted({0, k - 1}):
            assert_solution(lam[c].cpu().numpy(), ref[c], kappa, f"adjoint column {c}")
