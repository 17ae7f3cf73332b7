"""FP32 caplet plans on both sides of the rule that lets the caplet kernel draw its normals: the same theta
as the call without allocation (which always draws inside), on the sizes where the route changes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1408_5526_gb300 import inputs, rqmc  # noqa: E402


@pytest.mark.parametrize("seq, nf, N, M, launches", [
    ("philox", 20, 4099, 64, 2), ("philox", 20, 8193, 64, 3), ("philox", 21, 100, 2, 3),
    ("rasrap", 20, 4099, 32, 2), ("rasrap", 20, 4099, 40, 3), ("halton_rs", 21, 7, 1, 3),
    ("sobol_ds", 12, 4099, 30, 2), ("sobol_ds", 12, 4099, 34, 3), ("sobol_lms", 1, 1, 1, 2)])
def test_both_sides_price_the_same(seq, nf, N, M, launches):
    import torch
    lm, K = inputs.lmm_flat(nf), np.array([0.05])
    lm["vol"] = np.linspace(0.1, 0.2, nf)
    with rqmc.Plan.caplets(lm, K, N, M, seq, 5, prec="fp32") as p:
        assert p.launches() == launches
        a = p.execute().cpu().numpy()
    out = torch.empty(M * nf, dtype=torch.float64, device="cuda")
    rqmc.price_caplets_noalloc(lm, K, N, M, seq, 5, out, prec="fp32")
    # uniforms of bases p >= 7 differ by 1 to 2 ulp between the routes: the FP32 tolerance, 1e-4 of an accrual
    np.testing.assert_allclose(a, out.cpu().numpy(), rtol=1e-4, atol=1e-4 * 0.25 * 0.05)
