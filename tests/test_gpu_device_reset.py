"""A process that ends its device context (cudaDeviceReset) between calls: the staging
that synchronous calls keep is host memory of its own, so the calls after it work."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes
import numpy as np
import paper_2608_13110_gb300 as tb, workloads as W

lib, u8p, dp = tb._lib, ctypes.POINTER(ctypes.c_uint8), ctypes.POINTER(ctypes.c_double)
lib.tb_status_str(0)  # loads the library and with it the CUDA runtime
rt = ctypes.CDLL("libcudart.so.13")

def call(n, d, nb):
    c = W.random_circuit(n, d, None, nb, 3)
    plan, bits, out, ws = tb.Plan.from_circuit(c), np.ascontiguousarray(c.bits), np.zeros(2 * nb), ctypes.c_void_p()
    size = plan.workspace_bytes(nb)
    assert rt.cudaMalloc(ctypes.byref(ws), ctypes.c_size_t(size)) == 0
    rc = lib.tb_amplitudes(plan.handle, bits.ctypes.data_as(u8p), nb, ws, size, out.ctypes.data_as(dp), None)
    assert rc == 0, lib.tb_last_error()
    return out

cases = [(12, 8, 64), (10, 30, 2)]  # the narrow kernel and the passes
before = [call(*c) for c in cases]
assert rt.cudaDeviceReset() == 0
for c, want in zip(cases, before):
    for _ in range(2):
        assert np.array_equal(call(*c), want), c
print("same amplitudes")
"""


def test_calls_after_a_device_reset():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13110_gb300 import build as b
    b.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same amplitudes" in r.stdout, r.stdout + r.stderr
