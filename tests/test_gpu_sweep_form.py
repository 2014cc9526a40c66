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
    names = set()
    while not names:                                   # the first profile of a process comes back empty
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as pr:
            f()
            torch.cuda.synchronize()
        names = {e.name for e in pr.events()}
    return names


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


@pytest.mark.parametrize("layers,width,reach,dtype,k,blocks", [
    (200, 8, 1, 0, 1, True),        # narrow levels: 25 blocks of 64 rows against 200 levels in one CTA
    (200, 60, 1, 0, 1, False),      # 188 blocks against 200 levels of 3600 entries on the grid
    (200, 60, 1, 1, 1, False),
    (200, 60, 1, 0, 2, False),
    (200, 60, 1, 0, 16, True),      # a lane per entry: wide levels cost more than a block
    (100, 110, 1, 0, 16, False),    # 172 blocks against 100 levels, a CTA per row
    (400, 16, 8, 1, 16, True),      # 100 blocks against 400 levels
])
def test_form_follows_the_cost_of_blocks_and_levels(lsq, layers, width, reach, dtype, k, blocks):
    A, P = layered(lsq, layers, width, reach, coupling=0.1, precond_dtype=dtype)
    if k == 1:
        r = torch.ones(A.n, dtype=torch.float64, device="cuda")
        assert by_blocks(lambda: P.apply(r)) == blocks
    else:
        B = torch.ones(k, A.m, dtype=torch.float64, device="cuda")
        assert by_blocks(lambda: lsq.lsq_pcg_solve(A, P, B, lsq.opts(maxit=1, max_outer=1))) == blocks


def test_t0_builds_no_inverses(lsq):
    assert any("k_block_inverse" in x for x in kernels(lambda: layered(lsq, 200, 8, 1)))
    assert not any("k_block_inverse" in x for x in kernels(lambda: layered(lsq, 200, 8, 1, sweeps=0)))


def test_no_memory_for_the_inverses_leaves_the_row_forms(lsq):
    """3,000,000 rows in layers of 8 would take 3 GB of inverses; with 1.5 GB left the handle is built all
    the same and applies by rows."""
    n, width = 3000000, 8
    node = torch.arange(width, n, device="cuda")
    e = node.numel()
    rp = torch.cat([torch.arange(n, device="cuda"), n + 2 * torch.arange(e + 1, device="cuda")])
    ci = torch.cat([torch.arange(n, device="cuda"), torch.stack([node - width, node], 1).reshape(-1)]).to(torch.int32)
    va = torch.ones(n + 2 * e, dtype=torch.float64, device="cuda")
    va[n + 1::2] = -1.0
    A = lsq.Matrix(row_ptr=rp, col_idx=ci, vals=va, n=n)
    args = (torch.arange(A.m, dtype=torch.int32, device="cuda"),
            torch.full((A.m,), 1.0 / A.m, dtype=torch.float64, device="cuda"), torch.ones(n, dtype=torch.float64, device="cuda"))
    o = lsq.opts(precond_dtype=1)
    r = torch.randn(n, dtype=torch.float64, device="cuda")
    P = lsq.lsq_build_precond(A, *args, o)
    assert by_blocks(lambda: P.apply(r))
    E = P.apply(r)
    del P
    torch.cuda.synchronize()                           # the library gives back all but 1 GiB
    torch.cuda.empty_cache()
    fill, left = [], 3 << 29
    while torch.cuda.mem_get_info()[0] > left + (1 << 28):
        fill.append(torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda"))
    P = lsq.lsq_build_precond(A, *args, o)
    del fill
    assert not by_blocks(lambda: P.apply(r))
    assert float((P.apply(r) - E).norm() / E.norm()) <= 1e-10


def test_blocked_waits_run_out_then_recover(lsq):
    """With two polls a wait the blocked level chain and the blocked sweeps (one column, several) give
    up, report the timeout and leave the handle usable."""
    def limited(f):
        lsq.set_wait_limit(2)
        try:
            with pytest.raises(lsq.L.LsqError) as e:
                f()
            assert e.value.code == 6
        finally:
            lsq.set_wait_limit(0)

    kw = dict(layers=500, width=16, reach=2, coupling=0.1)     # 8000 rows, 32 dependencies: blocks for both
    A, P = layered(lsq, **kw)
    r = torch.randn(A.n, dtype=torch.float64, device="cuda")
    B = torch.randn(4, A.m, dtype=torch.float64, device="cuda")
    o = lsq.opts()
    apply, solve = lambda: P.apply(r), lambda: lsq.lsq_pcg_solve(A, P, B, o)
    assert by_blocks(apply) and by_blocks(solve)
    assert any("k_levels_blocked" in x for x in kernels(lambda: layered(lsq, **kw)))
    E, (X, info) = apply(), solve()
    limited(lambda: layered(lsq, **kw))
    limited(apply)
    limited(solve)
    assert torch.equal(apply(), E)
    X1, info = solve()
    assert torch.equal(X1, X) and all(info.converged == 1)
