"""FP32 log-Euler caplets on curves where some forwards are tiny (delta L of 2^-95): two adjacent forwards
share a reciprocal, and one that has been fixed must not disturb its alive neighbours.  The healthy
forwards' caplets agree with the FP64 plan within the 1e-4 of the FP32 parity tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1408_5526_gb300 import inputs, rqmc  # noqa: E402


def _model(nf, low, flat):
    lm = inputs.lmm_flat(nf)
    if not flat:
        lm["vol"] = 0.10 + 0.15 * (np.arange(nf) % 7) / 6.0
    tiny = np.zeros(nf, dtype=bool)
    tiny[{"even": slice(0, None, 2), "odd": slice(1, None, 2), "third": slice(2, None, 3)}[low]] = True
    lm["L0"][1:][tiny] = 1e-28
    return lm, ~tiny


@pytest.mark.parametrize("flat", [True, False])
@pytest.mark.parametrize("low", ["even", "odd", "third"])
@pytest.mark.parametrize("nf", [10, 33, 40, 66, 80, 97, 160])
def test_tiny_forwards_leave_their_neighbours_alone(nf, low, flat):
    import torch
    lm, ok = _model(nf, low, flat)
    K, N, M = np.array([0.05]), 1031, 2
    with rqmc.Plan.caplets(lm, K, N, M, "sobol_ds", 7, prec="fp64") as p:
        want = p.execute().cpu().numpy().reshape(M, nf)
    with rqmc.Plan.caplets(lm, K, N, M, "sobol_ds", 7, prec="fp32") as p:
        got = p.execute().cpu().numpy().reshape(M, nf)
    inside = torch.empty(M * nf, dtype=torch.float64, device="cuda")   # normals drawn in the kernel
    rqmc.price_caplets_noalloc(lm, K, N, M, "sobol_ds", 7, inside, prec="fp32")
    for th in (got, inside.cpu().numpy().reshape(M, nf)):
        assert np.isfinite(th).all()
        assert np.abs(th - want)[:, ok].max() <= 1e-4 * want[:, ok].max()
