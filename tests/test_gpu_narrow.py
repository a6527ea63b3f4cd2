"""Narrow boundaries (width <= 12, one CTA per bitstring) at every width: the
warp form (<= 7), the register windows with one CTA per SM and with several
(the window size differs), graph batches, both parities of the depth, and the
fewest rows (none, one, two between the first and the last)."""
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


@pytest.mark.parametrize("n", [2, 3, 4, 9, 10])
@pytest.mark.parametrize("h", range(1, 13))
def test_every_narrow_width(tb, oracle_mod, n, h):
    import torch
    for d in (2 * h, 2 * h - 1):
        if d < 2:
            continue
        u = W.random_unitaries(n, d, 100 * n + d)
        plan = tb.Plan(n, d, extra=[(q, t, u[t, q]) for t in range(d + 1) for q in range(n)])
        bits = np.random.default_rng(n + d).integers(0, 2, size=(400, n), dtype=np.uint8)
        ref = oracle_mod.sv_amplitudes(n, d, u, bits)
        few, many = plan.amplitudes(bits[:3]), plan.amplitudes(bits)
        assert np.linalg.norm(few - ref[:3]) <= TOL * np.linalg.norm(ref[:3])
        assert np.linalg.norm(many - ref) <= TOL * np.linalg.norm(ref)
        d_bits = torch.from_numpy(bits).cuda()
        d_out = torch.zeros((len(bits), 2), dtype=torch.float64, device="cuda")
        batch = tb.Batch([(plan, d_bits, d_out)])
        batch.launch()
        torch.cuda.synchronize()
        got = d_out.cpu().numpy()
        assert np.linalg.norm(got[:, 0] + 1j * got[:, 1] - ref) <= TOL * np.linalg.norm(ref)
