"""Narrow boundaries: an amplitude does not depend on how many bitstrings share the
call or on the entry point. Widths 11 and 12 run with another number of threads when
the bitstrings outnumber the SMs; the last row's sum keeps its grouping."""
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


@pytest.mark.parametrize("n,d", [(6, 16), (6, 19), (6, 21), (9, 22), (8, 23), (9, 24), (2, 22), (2, 24)])
def test_few_many_and_batch_give_the_same_bits(tb, n, d):
    import torch
    u = W.random_unitaries(n, d, 100 * n + d)
    u[:, n - 2, 1] *= 2.0 ** -9  # boundary entries from 1 to 2^-108: their FP64 sum is rounded
    plan = tb.Plan(n, d, extra=[(q, t, u[t, q]) for t in range(d + 1) for q in range(n)])
    bits = np.random.default_rng(n + d).integers(0, 2, size=(3200, n), dtype=np.uint8)
    many = plan.amplitudes(bits)
    few = np.concatenate([plan.amplitudes(bits[i:i + 100]) for i in range(0, len(bits), 100)])
    assert np.array_equal(few, many)
    d_bits, out = torch.from_numpy(bits).cuda(), torch.zeros((len(bits), 2), dtype=torch.float64, device="cuda")
    batch = tb.Batch([(plan, d_bits, out)])
    batch.launch()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.complex128)[:, 0], many)
