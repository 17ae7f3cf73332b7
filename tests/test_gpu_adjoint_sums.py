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
