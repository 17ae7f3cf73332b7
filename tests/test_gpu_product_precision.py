"""FP64 product integrand against extended precision (numpy's longdouble) on the same integer points.  A path's
product takes at most four roundings of 2^-53 a coordinate (factor, weight, two products) and the sums a
few more, whatever the weights: fixed point is used only where it rounds less."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1408_5526_gb300 import inputs, rqmc  # noqa: E402


def _denominators(seq, s):
    if seq in ("philox", "sobol_ds"):
        return [1 << 32] * s
    out, k = [], 2
    while len(out) < s:
        if all(k % p for p in range(2, k)):
            D = k
            while D * k < 1 << 64:
                D *= k
            out.append(D)
        k += 1
    return out


@pytest.mark.parametrize("seq, a, N, M", [
    ("philox", np.zeros(7), 1, 64), ("philox", np.zeros(2), 1, 64), ("sobol_ds", np.zeros(7), 2048, 16),
    ("sobol_ds", np.full(12, 1.0), 1024, 8), ("philox", np.full(5, 0.01), 3, 32), ("philox", np.full(3, 0.3), 1, 64),
    ("halton_rs", np.arange(1.0, 9.0), 4096, 32), ("rasrap", np.arange(1.0, 31.0), 100, 8),
    ("sobol_ds", np.arange(1.0, 41.0), 100, 8), ("halton_rs", np.full(2, 0.5), 1, 64), ("rasrap", np.full(9, 2.0), 1, 32)])
def test_product_rounds_no_more_than_fp64(seq, a, N, M):
    s = len(a)
    with rqmc.Plan.product(s, N, M, seq, 5, a) as p:
        got = p.execute().cpu().numpy()
    raw = rqmc.rqmc_points(s, N, M, seq, 5, transform="raw").cpu().numpy().view(np.uint64)
    f = np.ones((M, N), dtype=np.longdouble)
    for j, D in enumerate(_denominators(seq, s)):
        num = np.minimum(raw[:, j], np.uint64(D - 1) - raw[:, j]).astype(np.longdouble)
        f *= ((2 - 4 * ((num + np.longdouble(0.5)) / np.longdouble(D))) + np.longdouble(a[j])) / (1 + np.longdouble(a[j]))
    want = f.sum(axis=1) / N
    assert float(np.abs((got - want) / want).max()) <= (4 * s + 16) * 2.0**-53
