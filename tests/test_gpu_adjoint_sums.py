"""The adjoint's sums over many paths.  With zero volatilities every path is the same, so theta of a large
plan differs from theta of one path only by summation: per thread a column takes ppt / 2 <= 4 FP32 additions of
a pair of paths before it is emptied into float-float, 5 roundings of 2^-24 at most, 3e-7."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1408_5526_gb300 import inputs, rqmc  # noqa: E402


@pytest.mark.parametrize("nf,nK,N,M", [(3, 1, 130, 3), (10, 1, (1 << 18) + 3, 64), (41, 3, 50001, 40), (10, 2, 99999, 70)])
def test_equal_paths_sum_without_loss(nf, nK, N, M):
    lm = inputs.lmm_flat(nf)
    lm["vol"] = np.zeros(nf)
    lm["L0"] = 0.05 * (1 + 0.1 * np.arange(nf + 1) / nf)
    K, w = np.linspace(0.03, 0.04, nK), np.linspace(0.5, 1.5, nf * nK)
    rows = []
    for n, m in ((1, 1), (N, M)):
        with rqmc.Plan.adjoint(lm, K, w, n, m, "philox", 1) as p:
            out = p.execute().cpu().numpy().reshape(m, -1)
        rows.append(np.delete(out, np.s_[1 + nf:1 + 2 * nf], axis=1))   # value, deltas, prices (vegas follow the normals)
    np.testing.assert_allclose(rows[1], np.broadcast_to(rows[0], rows[1].shape), rtol=3e-7)


@pytest.mark.parametrize("nf, d, N, M, split", [(3, 1, 70001, 200, 33333), (5, 2, 9001, 40, 4500), (42, 2, 20003, 30, 1)])
def test_units_of_every_size_and_their_partly_filled_last_one(nf, d, N, M, split):
    """Two plans over the halves of a point range add up to the plan over all of it: the same paths in units
    of other sizes, whose last ones leave threads and warps without a path."""
    lm = inputs.lmm_two_factor(nf, seed=2) if d == 2 else inputs.lmm_flat(nf)
    K, w = np.array([0.045, 0.05]), np.linspace(0.5, 1.5, 2 * nf)
    th = []
    for off, n in ((0, N), (0, split), (split, N - split)):
        with rqmc.Plan.adjoint(lm, K, w, n, M, "philox", 4, offset=off) as p:
            th.append(n * p.execute().cpu().numpy())
    whole, parts = th[0], th[1] + th[2]
    rows = np.abs(whole.reshape(M, -1))
    # the sums round at 3e-7 of their terms' sizes; vegas cancel among theirs: the Greeks' 1e-4
    assert np.abs(whole - parts).max() <= 1e-4 * rows.max()
    np.testing.assert_allclose(parts.reshape(M, -1)[:, 0], whole.reshape(M, -1)[:, 0], rtol=1e-6)
    np.testing.assert_allclose(parts.reshape(M, -1)[:, 1:1 + nf], whole.reshape(M, -1)[:, 1:1 + nf], rtol=1e-4)
    np.testing.assert_allclose(parts.reshape(M, -1)[:, 1 + nf:1 + 2 * nf], whole.reshape(M, -1)[:, 1 + nf:1 + 2 * nf], rtol=1e-4,
                               atol=1e-4 * rows[:, 1 + nf:1 + 2 * nf].max())
