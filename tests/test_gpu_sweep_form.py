"""Which form the sparse sweeps take and what it computes, on matrices whose A^T A has layers of
nodes that depend on the layer before: the depth and the length of the rows are the test's choice."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def layered(lsq, layers, width, reach, coupling=0.5, seed=0, **kw):
    """(Matrix, Precond): every node joined with all nodes of the `reach` layers before its own; one row
    of A per node and per edge, every row drawn once, so that M = A^T A exactly."""
    rng = np.random.default_rng(seed)
    n = layers * width
    node, back, at = (x.reshape(-1) for x in np.meshgrid(np.arange(n), np.arange(1, reach + 1), np.arange(width),
                                                         indexing="ij"))
    keep = node // width >= back
    node, other = node[keep], ((node // width - back) * width + at)[keep]
    e = node.size
    w = coupling * rng.uniform(0.5, 1.0, e)
    rows = np.concatenate([np.arange(n), n + np.arange(e), n + np.arange(e)])
    cols = np.concatenate([np.arange(n), node, other])
    vals = np.concatenate([rng.uniform(0.5, 2.0, n), w, -w])
    order = np.lexsort((cols, rows))
    m = n + e
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    cuda = lambda x, t: torch.from_numpy(np.ascontiguousarray(x, dtype=t)).cuda()
    A = lsq.Matrix(row_ptr=cuda(rp, np.int64), col_idx=cuda(cols[order], np.int32), vals=cuda(vals[order], np.float64), n=n)
    P = lsq.lsq_build_precond(A, torch.arange(m, dtype=torch.int32, device="cuda"),
                              torch.full((m,), 1.0 / m, dtype=torch.float64, device="cuda"),
                              torch.ones(n, dtype=torch.float64, device="cuda"), lsq.opts(**kw))
    return A, P


def kernels(f):
    """Names of the kernels that f launches."""
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as pr:
        f()
        torch.cuda.synchronize()
    return {e.name for e in pr.events()}


def by_blocks(f):
    return any("k_sweep_blocked" in k for k in kernels(f))


@pytest.fixture
def form(lsq):
    yield lsq.set_sweep_form
    lsq.set_sweep_form(0)


@pytest.mark.parametrize("k", [2, 4, 7])
def test_fp32_m_summed_in_fp64_uses_fp64_inverses(lsq, form, k):
    """Rows of 32 dependencies (a lane per entry, FP64 sums) by blocks against the row form, for a nearly
    diagonal M: one iteration from zero is alpha times one forward and one backward sweep, and the two
    forms' entries differ by the roundings of a diagonal's reciprocal and two products in each sweep and
    of alpha, 9 in all.  (Inverses kept to 48 bits are off by up to 2^-49 a sweep.)"""
    A, P = layered(lsq, 40, 16, 2, coupling=1e-9, precond_dtype=1)
    B = torch.randn(k, A.m, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    o = lsq.opts(maxit=1, max_outer=1, precond_dtype=1)
    solve = lambda: lsq.lsq_pcg_solve(A, P, B, o)[0]
    assert by_blocks(solve)
    X0 = solve()
    form(1)
    assert not by_blocks(solve)
    X1 = solve()
    assert float(((X0 - X1).abs() / X1.abs()).max()) <= 9 * 2.0 ** -53
