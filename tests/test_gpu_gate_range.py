"""Narrow boundaries (widths 1 to 12) with one-qubit gates of very different magnitude:
`extra` takes any 2x2 matrix, and a power of two on one gate only scales the
amplitudes, wherever in a row the gate sits and whatever its neighbours bring."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the library's bar for complex64, as in test_gpu_parity.py
BIG = 80    # 2^80 twice, or against 2^-80 twice, is beyond FP32's range


@pytest.fixture(scope="module")
def tb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13110_gb300 import build as b
    b.build()
    import paper_2608_13110_gb300 as mod
    return mod


def _check(tb, oracle_mod, n, d, scaled):
    """scaled: (qubit, slot, exponent) of the gates multiplied by a power of two."""
    import torch
    u = W.random_unitaries(n, d, 10 * n + d)
    bits = np.random.default_rng(d).integers(0, 2, size=(400, n), dtype=np.uint8)
    ref = oracle_mod.sv_amplitudes(n, d, u, bits) * 2.0 ** sum(e for _, _, e in scaled)
    g = u.copy()
    for q, t, e in scaled:
        g[t, q] *= 2.0 ** e
    plan = tb.Plan(n, d, extra=[(q, t, g[t, q]) for t in range(d + 1) for q in range(n)])
    d_bits, out = torch.from_numpy(bits).cuda(), torch.zeros((len(bits), 2), dtype=torch.float64, device="cuda")
    batch = tb.Batch([(plan, d_bits, out)])
    batch.launch()
    torch.cuda.synchronize()
    for got, want in ((plan.amplitudes(bits[:3]), ref[:3]), (plan.amplitudes(bits), ref),
                      (out.cpu().numpy().view(np.complex128)[:, 0], ref)):
        assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want), scaled


# Step p of an absorbed row holds slot 2p + 1; odd rows walk p upwards, even rows
# downwards. A gate at the row's first step against one at every later step.
@pytest.mark.parametrize("h", [4, 7, 8, 9, 10, 11, 12])
@pytest.mark.parametrize("sign", [1, -1])
def test_opposite_magnitudes_within_a_row(tb, oracle_mod, h, sign):
    for p in range(1, h):
        _check(tb, oracle_mod, 5, 2 * h, [(1, 1, sign * BIG), (1, 2 * p + 1, -sign * BIG)])
        _check(tb, oracle_mod, 5, 2 * h, [(2, 2 * h - 1, sign * BIG), (2, 2 * (h - 1 - p) + 1, -sign * BIG)])


# The last step of one row and the first of the next.
@pytest.mark.parametrize("h", [4, 7, 8, 9, 10, 11, 12])
@pytest.mark.parametrize("sign", [1, -1])
def test_equal_magnitudes_at_a_turn(tb, oracle_mod, h, sign):
    _check(tb, oracle_mod, 5, 2 * h, [(1, 2 * h - 1, sign * BIG), (2, 2 * h - 1, sign * BIG)])  # top
    _check(tb, oracle_mod, 5, 2 * h, [(2, 1, sign * BIG), (3, 1, sign * BIG)])                  # bottom
