"""The batch's tile products at the edges of their shares: column counts at every padded width
(1, 2, 4, 8, 16), n around the chunks of four columns and the shares of 32, m around the tiles
of 32 rows, NaN in A's padding.  The answer minimises ||Ax - b||: the normal equations hold to the tolerance
of the solve (1e-10 of ||D^-1 A^T b||, the quantity it stops on, computed here in FP64; a factor 2 for
the double-float residual behind its own test)."""
import numpy as np
import pytest

import workloads as W
from test_gpu_batch import _opts, _problem

pytestmark = pytest.mark.gpu
SHAPES = [(97, 1), (130, 3), (131, 4), (193, 5), (320, 31), (415, 33), (640, 64), (1003, 127), (1601, 129), (3100, 255), (3211, 256)]


@pytest.mark.parametrize("cluster", [1, 4])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 7, 8, 13, 16])
def test_batch_tile_edges(lsq, k, cluster):
    rng = np.random.default_rng(k)
    mats = [{"kind": "dense", "A": rng.standard_normal((m, n))} for m, n in SHAPES]
    prs = [_problem(lsq, mt, 40 + i, k, 1e-2) for i, mt in enumerate(mats)]
    o = _opts(lsq)
    bt = lsq.Batch([(pr["T"], pr["n"], pr["P"], pr["B"]) for pr in prs], o)
    bt.set_cluster(cluster)
    bt.solve()
    for pr, X, info in zip(prs, bt.X, bt.info()):
        A, b, x = pr["seen"]["A"], pr["b"], X.cpu().numpy().reshape(k, -1)
        d = np.linalg.norm(A, axis=0)
        for c in range(k):
            r = np.linalg.norm(A.T @ (b[c] - A @ x[c]) / d) / np.linalg.norm(A.T @ b[c] / d)
            assert info.converged[c] == 1 and r <= 2 * o.tol, (A.shape, c, r)
