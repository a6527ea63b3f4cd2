"""Narrow plans (widths 1 to 12) in a workspace that is aligned to 8 bytes only, such as a
slice of a larger buffer: the tables hold 8-byte values, and no entry asks for more."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13110_gb300 import build as b
    b.build()
    import paper_2608_13110_gb300 as mod
    return mod


@pytest.mark.parametrize("h", range(1, 13))
def test_workspace_aligned_to_8_bytes(tb, h):
    import torch
    for d in (2 * h, 2 * h - 1):
        if d < 2:
            continue
        c = W.random_circuit(9, d, None, 300, d)
        plan = tb.Plan.from_circuit(c)
        want = plan.amplitudes(c.bits)
        ws = torch.empty(plan.workspace_bytes(300) + 8, dtype=torch.uint8, device="cuda")[8:]
        assert ws.data_ptr() % 16 == 8
        assert np.array_equal(plan.amplitudes(c.bits, ws=ws), want)
        plan.upload(ws)
        bits, out = torch.from_numpy(c.bits).cuda(), torch.zeros((300, 2), dtype=torch.float64, device="cuda")
        plan.amplitudes_device(bits, ws, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().view(np.complex128)[:, 0], want)
        # a graph batch in such a workspace, through the C interface
        out.zero_()
        item = (tb._BatchItem * 1)(tb._BatchItem(plan.handle, bits.data_ptr(), 300, out.data_ptr()))
        need = tb._lib.tb_batch_workspace_bytes(ctypes.byref(item), 1)
        ws = torch.empty(need + 8, dtype=torch.uint8, device="cuda")[8:]
        batch, st = ctypes.c_void_p(), torch.cuda.current_stream().cuda_stream
        assert tb._lib.tb_batch_create(ctypes.byref(item), 1, ws.data_ptr(), need, 0, st, ctypes.byref(batch)) == tb.TB_OK
        assert tb._lib.tb_batch_launch(batch, st) == tb.TB_OK
        torch.cuda.synchronize()
        tb._lib.tb_batch_destroy(batch)
        assert np.array_equal(out.cpu().numpy().view(np.complex128)[:, 0], want)
