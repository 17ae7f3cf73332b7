"""Default launch shapes by plan size: each side of a rule gives theta of the smallest shape to summation
order, and FP32 mortgage plans that the run kernel cannot take keep the shape of the kernel they run."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1408_5526_gb300 import inputs, rqmc  # noqa: E402


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("N, M", [(1, 1), (4099, 32), (7001, 50), (7001, 300), (20011, 100)])
def test_product_shapes(N, M, prec):
    with rqmc.Plan.product(5, N, M, "rasrap", 3, inputs.product_weights(5), prec=prec) as p:
        a = p.execute().cpu().numpy()
        p.set_launch(threads=32, paths_per_thread=1)
        b = p.execute().cpu().numpy()
    # a tile's FP32 warp totals are added with compensation: one rounding of 2^-24 each way; up to 30 FP64 sums in line
    np.testing.assert_allclose(a, b, rtol=4e-15 if prec == "fp64" else 2.4e-7)


@pytest.mark.parametrize("seq, months, offset, shape", [
    ("sobol_ds", 60, 13, (256, 4)), ("sobol_ds", 1500, 255, (256, 4)), ("rasrap", 1500, 0, (256, 2)),
    ("sobol_ds", 60, 512, None), ("philox", 1500, 13, None), ("rasrap", 60, 13, None)])
def test_mbs_shape_of_the_kernel_that_runs(seq, months, offset, shape):
    mb, N, M = inputs.mbs_paper(months), 8191, 64
    with rqmc.Plan.mbs(mb, N, M, seq, 3, prec="fp32", offset=offset) as p:
        got = p.launch_shape()
        assert got == shape if shape else got[1] == 8
        a = p.execute().cpu().numpy()
    with rqmc.Plan.mbs(mb, N, M, seq, 3, prec="fp64", offset=offset) as p:
        b = p.execute().cpu().numpy()
    np.testing.assert_allclose(a, b, rtol=1e-5)   # the FP32 tolerance of the parity tests
