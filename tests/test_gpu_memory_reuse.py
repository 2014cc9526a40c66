"""Scratch comes back from earlier calls with whatever they left in it: a solve after one whose
buffers were full of NaN must give the bits of a solve on fresh memory."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,k", [("dense", 1), ("dense", 3), ("csr", 1), ("csr", 3), ("csr_persistent", 3)])
def test_solve_does_not_depend_on_what_scratch_holds(lsq, kind, k):
    mat = W.gaussian_dense(3000, 60, 3) if kind == "dense" else W.sparse_random(20000, 300, 8, 3)
    Mx, keep, seen = to_device(lsq, mat)
    o = lsq.opts(seed=3, device_loop=1 if kind == "csr_persistent" else 0)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    P = lsq.lsq_build_precond(Mx, idx, p, d, o)
    xs, b = W.rhs_for(seen, k, 1e-3, 4)
    if k > 1:
        b[1] = 0.0                                     # a column that never iterates
    B = torch.from_numpy(b).cuda()
    X0, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    assert np.all(info.converged == 1)
    bad = B.clone()
    bad[0, 5] = float("nan")
    with pytest.raises(lsq.L.LsqError):
        lsq.lsq_pcg_solve(Mx, P, bad.expand(k, -1).contiguous() * float("nan"), o)
    X1, info = lsq.lsq_pcg_solve(Mx, P, B, o)
    assert torch.equal(X0, X1) and np.all(info.converged == 1)
