"""A_s^T A_s of a dense matrix, entry by entry, against extended precision for draws that the test
chooses itself."""
import numpy as np
import pytest
import torch

from helpers import to_device

pytestmark = pytest.mark.gpu


def _normal_matrix(lsq, A, idx, p, d):
    """(M, the exact one in extended precision, the sums of magnitudes of its terms)"""
    Mx, keep, seen = to_device(lsq, {"kind": "dense", "A": A})
    cuda = lambda x, t: torch.from_numpy(np.ascontiguousarray(x, dtype=t)).cuda()
    P = lsq.lsq_build_precond(Mx, cuda(idx, np.int32), cuda(p, np.float64), cuda(d, np.float64), lsq.opts())
    X = A[idx].astype(np.longdouble) / d.astype(np.longdouble)
    g = 1 / (np.longdouble(len(idx)) * p.astype(np.longdouble))
    return P.M().cpu().numpy(), X.T @ (g[:, None] * X), np.abs(X).T @ (g[:, None] * np.abs(X))


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -300])
def test_columns_without_a_draw_are_exactly_zero(lsq, scale):
    """Columns that are zero in every drawn row (an undrawn part of the identity, an empty column), at
    both ends of a tile and inside it."""
    rng = np.random.default_rng(1)
    m, n = 600, 130
    A = rng.standard_normal((m, n)) * scale
    zero = [0, 63, 64, 100, 129]
    A[:, zero] = 0.0
    A[m - 1, zero[:3]] = scale                         # a row that no draw takes
    idx = rng.integers(0, m - 1, 400)
    M, exact, mag = _normal_matrix(lsq, A, idx, np.full(400, 1.0 / m), np.full(n, scale))
    for j in zero:
        assert M[j, j] == 1.0
        assert np.all(np.delete(M[j], j) == 0.0) and np.all(np.delete(M[:, j], j) == 0.0)


@pytest.mark.parametrize("kind", ["even", "spike1e-5", "spike1e-8", "one_wide", "tiny"])
@pytest.mark.parametrize("n,s", [(1, 40), (63, 900), (65, 3000), (130, 257), (3, 100000)])
def test_every_entry_is_as_accurate_as_an_fp64_product(lsq, n, s, kind):
    """Columns whose entries lie far below one that stands out (each in a row of its own), one such
    column among others, a column far below its scale, and columns without any: every entry of M within
    the a-priori bound of an FP64 product, s + 6 roundings (scale, root, products and sums) of the sum of
    its terms' magnitudes."""
    rng = np.random.default_rng(n + s)
    m = 2 * n + 500
    A = rng.standard_normal((m, n))
    wide = range(n) if kind.startswith("spike") else [n // 2]
    if kind != "even":
        small = 1e-5 if kind == "spike1e-5" else 1e-8
        if kind == "tiny":
            small = 2.0 ** -1000
        for j in wide:
            A[:, j] *= small
            A[j] = 0.0
            A[j, j] = 1.0
    idx = rng.integers(n if kind == "tiny" else 0, m, s)
    if kind != "tiny":
        idx[:n] = np.arange(n)[:s]                     # the rows that stand out are drawn
    w = rng.uniform(0.5, 2.0, m)
    d = rng.uniform(0.5, 2.0, n)
    if kind == "tiny":
        d[n // 2] = 2.0 ** -400
    M, exact, mag = _normal_matrix(lsq, A, idx, (w / w.sum())[idx], d)
    fixed = np.diag(M) == 1.0                          # M_jj that underflows counts as zero and is replaced
    assert np.array_equal(M, M.T)
    err = np.abs(M - exact)
    err[fixed & (np.diag(mag) < 1e-300), fixed & (np.diag(mag) < 1e-300)] = 0.0
    assert np.all(err <= (s + 6) * 2.0 ** -53 * mag)
