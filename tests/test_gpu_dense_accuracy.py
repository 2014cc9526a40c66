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
