"""FP32 log-Euler caplets whose normals are drawn inside the caplet kernel, over the register buckets that
small plans do not reach (more than 40 forwards, as in calls without allocation and plans whose
normals exceed their buffer's cap), against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1408_5526_gb300 import inputs

JK = inputs.joe_kuo_table()
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nf", [1, 16, 17, 40, 41, 66, 80, 81, 97, 160])
@pytest.mark.parametrize("flat", [True, False])
def test_caplets32_normals_inside(nf, flat):
    import torch
    from paper_1408_5526_gb300 import rqmc
    lm = inputs.lmm_flat(nf, vol=0.15)
    lm["L0"] = np.linspace(0.04, 0.06, nf + 1)
    if not flat:
        lm["vol"] = np.linspace(0.1, 0.2, nf)
        lm["vol"][nf // 2] = 0.0 if nf > 2 else 0.1
    K, M = np.array([0.045, 0.05, 0.055]), 2
    out = torch.empty(M * nf * 3, dtype=torch.float64, device="cuda")
    for seq in (O.RASRAP, O.SOBOL_DS, O.PHILOX):
        for N in (1, 33, 1031):
            th_o = O.lmm_caplets(O.Sequence(seq, nf, M, 17, joe_kuo=JK), lm, K, N)
            rqmc.price_caplets_noalloc(lm, K, N, M, seq, 17, out, prec="fp32")
            th = out.cpu().numpy().reshape(th_o.shape)
            # the tolerance of test_gpu_caplets32.py: 1e-4 of the caplet or of one accrual 0.25 * 0.05
            assert np.all(np.abs(th - th_o) <= 1e-4 * np.maximum(np.abs(th_o), 0.25 * 0.05)), (N, seq)
