"""How the columns of a dense solve share the grid: matrices larger than L2 one after the other (each
column then has the bits of a solve of its own), smaller ones side by side with every group taking
the next column when it is done."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import assert_solution, to_device

pytestmark = pytest.mark.gpu


def _handle(lsq, mat, dtype="f64"):
    Mx, keep, seen = to_device(lsq, mat, dtype, with_f64=dtype == "f32", ld_pad=(-mat["A"].shape[1]) % 4)
    o = lsq.opts(seed=5, max_outer=30, inner_tol=1e-4 if dtype == "f32" else 0.0)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    return Mx, keep, seen, o, d, lsq.lsq_build_precond(Mx, idx, p, d, o)


@pytest.mark.parametrize("dtype,m", [("f64", 150000), ("f32", 300000)])
def test_columns_of_a_large_matrix_have_the_bits_of_single_solves(lsq, dtype, m):
    Mx, keep, seen, o, d, P = _handle(lsq, W.gaussian_dense(m, 120, 3), dtype)
    B = torch.randn(3, m, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    B[1] = 0.0
    X, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    for c in range(3):
        x1, i1 = lsq.lsq_pcg_solve(Mx, P, B[c], o)
        assert torch.equal(X[c], x1) and info.iters[c] == i1.iters[0]


@pytest.mark.parametrize("slow", [[0], [16, 32], [0, 16, 32], list(range(1, 33, 2))])
def test_groups_take_the_next_column(lsq, slow):
    """33 columns, some of them zero (done at once): whichever group takes a column, it comes out as it
    does with no zero columns around it, to the bit, since all groups are the same size."""
    Mx, keep, seen, o, d, P = _handle(lsq, W.gaussian_dense(5000, 130, 7))
    B = torch.randn(33, 5000, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    full, fi = lsq.lsq_pcg_solve(Mx, P, B, o)
    Z = torch.zeros_like(B)
    Z[slow] = B[slow]
    X, info = lsq.lsq_pcg_solve(Mx, P, Z, o)
    assert all(info.converged == 1)
    for c in range(33):
        if c in slow:
            assert torch.equal(X[c], full[c]) and info.iters[c] == fi.iters[c]
        else:
            assert info.iters[c] == 0 and torch.all(X[c] == 0.0)
    kappa = np.linalg.cond(seen["A"] / d.cpu().numpy())
    assert_solution(X[slow[0]].cpu().numpy(), np.linalg.lstsq(seen["A"], B[slow[0]].cpu().numpy(), rcond=None)[0], kappa,
                    "column %d" % slow[0])


def test_barriers_of_the_groups_run_out_then_recover(lsq):
    """With two polls a wait the barriers of several groups give up, the call reports the timeout, and the
    next one gives the same bits as before."""
    Mx, keep, seen, o, d, P = _handle(lsq, W.gaussian_dense(5000, 130, 7))
    B = torch.randn(8, 5000, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    X, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    lsq.set_wait_limit(2)
    try:
        with pytest.raises(lsq.L.LsqError) as e:
            lsq.lsq_pcg_solve(Mx, P, B, o)
        assert e.value.code == 6
    finally:
        lsq.set_wait_limit(0)
    X1, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    assert torch.equal(X1, X) and all(info.converged == 1)
