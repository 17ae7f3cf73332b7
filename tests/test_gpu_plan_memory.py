"""FP32 caplet and adjoint plans without memory for their normals buffer draw the normals in the path kernel
and price the same.  A child process gives its device a memory pool of 32 MiB, so that the buffer (42 MB
and more) cannot be had while the GPU itself stays empty."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes as C, sys
import numpy as np, torch
torch.zeros(1, device="cuda")
from paper_1408_5526_gb300 import inputs, rqmc
rqmc.load()
rt = C.CDLL("libcudart.so.13")

class Props(C.Structure):   # cudaMemPoolProps
    _fields_ = [("alloc", C.c_int), ("handles", C.c_int), ("loc", C.c_int), ("dev", C.c_int), ("sec", C.c_void_p),
                ("max_size", C.c_size_t), ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]

lm, K, N, M = inputs.lmm_flat(40), np.array([0.05]), 4099, 64
lm["vol"] = np.linspace(0.1, 0.2, 40)

def price():
    out = []
    for seq in ("sobol_ds", "rasrap"):
        with rqmc.Plan.caplets(lm, K, N, M, seq, 3, prec="fp32") as p:
            out.append((p.launches(), p.execute().cpu().numpy()))
        with rqmc.Plan.adjoint(lm, K, np.ones(40), N, M, seq, 3) as p:
            out.append((p.launches(), p.execute().cpu().numpy()))
    return out

full = price()
pool, props = C.c_void_p(), Props(1, 0, 1, 0, None, 32 << 20, 0)
assert rt.cudaMemPoolCreate(C.byref(pool), C.byref(props)) == 0
assert rt.cudaDeviceSetMemPool(0, pool) == 0
small = price()
assert [n for n, _ in full] == [3, 3, 3, 3] and [n for n, _ in small] == [2, 2, 2, 2], ([n for n, _ in full], [n for n, _ in small])
for i, ((_, a), (_, b)) in enumerate(zip(full, small)):
    # Sobol' normals are the same bits.  Rasrap's uniforms differ by 1 to 2 ulp, so that a path within FP32
    # rounding of a strike may take the other branch, which moves a delta or vega by w delta D / N:
    # values and prices only.
    if i == 3:
        a, b = (np.delete(x.reshape(M, -1), np.s_[1:81], axis=1) for x in (a, b))
    np.testing.assert_allclose(b, a, rtol=1e-4, atol=1e-4 * np.abs(a).min() + 1e-7)
print("same")
"""


def test_plans_price_without_a_normals_buffer():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("same"), r.stdout + r.stderr
