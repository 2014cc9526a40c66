"""Dense preconditioner setup at the edges of its tiles: A_s^T A_s on the tensor cores (64-column
tiles, 128-draw sums) and the materialised operator (32-row blocks, 1 to 4 columns per CTA)
against the oracle, with the bars of the same quantities elsewhere: entries of M at rtol 1e-12
(sums in another order), the operator at 1e-12 of literal Alg. 3 on well-conditioned matrices."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import rel, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("n,sweeps", [(1, 1), (2, 2), (31, 1), (32, 2), (33, 1), (63, 1), (64, 2), (65, 1), (97, 3),
                                      (153, 1), (305, 2), (457, 1)])
def test_dense_build_at_tile_edges(lsq, orc, n, sweeps, dtype):
    mat = W.gaussian_dense(max(8 * n, 50), n, n + 5)
    Mx, keep, seen = to_device(lsq, mat, dtype)
    o = lsq.opts(seed=n, sweeps=sweeps)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    P = lsq.lsq_build_precond(Mx, idx, p, d, o)
    smp = orc.Sample(seen, seed=n)
    Mo = orc.SampledM(smp)
    Mg, Md = P.M().cpu().numpy(), Mo.dense()
    assert np.array_equal(Mg, Mg.T)
    np.testing.assert_allclose(Mg, Md, rtol=1e-12, atol=1e-13 * np.abs(Md).max())
    R = np.random.default_rng(n).standard_normal((2, n))
    E = P.apply(torch.from_numpy(R).cuda()).cpu().numpy()
    for c in range(2):
        assert rel(E[c], orc.sgs_apply(Mo, R[c], sweeps)) <= 1e-12


@pytest.mark.parametrize("scale", [2.0 ** -400, 2.0 ** 400])
@pytest.mark.parametrize("sampling", [0, 1])
def test_normal_matrix_scales_and_densities(lsq, orc, scale, sampling):
    """Columns of very different sizes, rows of very different norms, both densities: the digits
    are cut per column after the scaling, so M keeps its relative accuracy."""
    rng = np.random.default_rng(3)
    A = rng.standard_normal((3000, 70)) * np.where(rng.random((3000, 1)) < 0.05, 1.0, 1e-3)
    A[:, 7] *= scale
    A[:, 13] = 0.0
    mat = {"kind": "dense", "A": A}
    Mx, keep, seen = to_device(lsq, mat)
    o = lsq.opts(seed=4, sampling=sampling)
    idx, p, d = lsq.lsq_sample_rows(Mx, o)
    P = lsq.lsq_build_precond(Mx, idx, p, d, o)
    smp = orc.Sample(seen, seed=4, sampling="uniform" if sampling else "norm2")
    Md = orc.SampledM(smp).dense()
    np.testing.assert_allclose(P.M().cpu().numpy(), Md, rtol=1e-12, atol=1e-13 * np.abs(Md).max())
