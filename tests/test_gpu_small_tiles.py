"""Small tiles of the boundary passes (few bitstrings of a narrow boundary) against
whole tiles (the same bitstring in a batch that fills the device): the same steps
in the same order, so the amplitudes are the same bits, and both against the
state vector. The schedules use every window size that has small tiles, at bit 0
and above it, in forward, reversed, turn, first and last passes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the library's bar for complex64, as in test_gpu_parity.py


@pytest.fixture(scope="module")
def tb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13110_gb300 import build as b
    b.build()
    import paper_2608_13110_gb300 as mod
    return mod


# n, d, window / bottom / top bits: middle windows of 9, 8, 7, 6 and 5 bits at
# width 19, then turns of 5 to 10 bits; odd and even numbers of rows
SCHEDULES = [(6, 38, 9, 6, 6), (7, 38, 8, 6, 7), (6, 38, 7, 7, 7), (7, 37, 6, 8, 7), (6, 38, 5, 9, 7),
             (7, 26, 5, 5, 9), (6, 26, 5, 9, 5), (7, 26, 5, 6, 8), (6, 28, 10, 5, 10), (7, 36, 10, 10, 9),
             (6, 27, 5, 8, 7), (8, 30, 0, 0, 0), (9, 33, 0, 0, 0)]


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("n,d,wb,bb,tt", SCHEDULES)
def test_small_tiles_equal_whole_tiles(tb, oracle_mod, n, d, wb, bb, tt, dense):
    c = W.random_circuit(n, d, None, 500, 100 * n + d)
    opts = dict(window_bits=wb, bottom_bits=bb, top_bits=tt)
    if dense:
        u = W.random_unitaries(n, d, 7 * n + d)
        plan = tb.Plan(n, d, extra=[(q, t, u[t, q]) for t in range(d + 1) for q in range(n)], **opts)
    else:
        u = oracle_mod.circuit_gates(c)
        plan = tb.Plan.from_circuit(c, **opts)
    ref = oracle_mod.sv_amplitudes(n, d, u, c.bits)
    many = plan.amplitudes(c.bits)
    assert np.linalg.norm(many - ref) <= TOL * np.linalg.norm(ref)
    for i, nb in ((0, 1), (5, 2), (17, 3)):
        few = plan.amplitudes(c.bits[i:i + nb])
        assert np.array_equal(few, many[i:i + nb])
