"""rqmc_plan_launches against the kernels of one execute: FP64 log-Euler caplets in fixed point launch the
fixed-point kernel, the guarded floating-point one and theta; outside fixed point two."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1408_5526_gb300 import inputs, rqmc  # noqa: E402


def _kernels(plan):
    """Nodes of the graph that one execute is captured into: its kernels, nothing else."""
    import torch
    out = torch.empty(plan.output_size(), dtype=torch.float64, device="cuda")
    plan.execute(out)   # kernel attributes are set outside the capture
    torch.cuda.synchronize()
    rt, st = C.CDLL("libcudart.so.13"), torch.cuda.Stream()
    graph, n = C.c_void_p(), C.c_size_t()
    assert rt.cudaStreamBeginCapture(C.c_void_p(st.cuda_stream), 2) == 0   # relaxed
    plan.execute(out, stream=st)
    assert rt.cudaStreamEndCapture(C.c_void_p(st.cuda_stream), C.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, C.byref(n)) == 0
    rt.cudaGraphDestroy(graph)
    return n.value


@pytest.mark.parametrize("form, count", [("fixed", 3), ("wide vol", 2), ("256 threads", 2), ("euler", 2), ("fp32", 2),
                                         ("fp32 buffer", 3), ("product", 1), ("mbs", 2), ("adjoint", 3), ("adjoint philox", 2)])
def test_plan_launches_counts_the_kernels(form, count):
    lm, K, N, M, seq = inputs.lmm_flat(12), np.array([0.05]), 1024, 2, "sobol_ds"
    if form == "product":
        p = rqmc.Plan.product(3, N, M, seq, 1, inputs.product_weights(3))
    elif form == "mbs":
        p = rqmc.Plan.mbs(inputs.mbs_paper(24), N, M, seq, 1, prec="fp32")
    elif form.startswith("adjoint"):
        p = rqmc.Plan.adjoint(lm, K, np.ones(12), N, M, "philox" if "philox" in form else seq, 1)
    else:
        if form == "wide vol":
            lm = inputs.lmm_flat(12, delta=1.0, vol=1.2)
        if form == "euler":
            lm = inputs.lmm_flat(12, scheme=1)
        if form == "fp32 buffer":
            lm = inputs.lmm_flat(60)
        p = rqmc.Plan.caplets(lm, K, N, M, seq, 1, prec="fp32" if form.startswith("fp32") else "fp64")
        if form == "256 threads":
            p.set_launch(threads=256)
    with p:
        assert p.launches() == count == _kernels(p)
