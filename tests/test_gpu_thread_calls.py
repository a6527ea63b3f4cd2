"""Synchronous calls from many host threads: the staging that a call borrows belongs
to no thread, so a thread that ends waits for nobody else's device work, and calls
beyond the number of staging blocks give the same amplitudes."""
import os
import threading
import time

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


def test_thread_that_ends_leaves_the_device_alone(tb):
    import torch
    small, wide = W.random_circuit(12, 8, None, 64, 1), W.random_circuit(30, 52, None, 1, 3)
    ps, pw = tb.Plan.from_circuit(small), tb.Plan.from_circuit(wide)
    ws, ww = ps.alloc_workspace(64), pw.alloc_workspace(1)
    want = ps.amplitudes(small.bits, ws=ws)
    pw.upload(ww)
    bits, out = torch.from_numpy(wide.bits).cuda(), torch.zeros((1, 2), dtype=torch.float64, device="cuda")
    side, busy = torch.cuda.Stream(), torch.cuda.Stream()
    done, got, tid = torch.cuda.Event(), [], []

    def call():
        torch.cuda.set_device(0)
        tid.append(threading.get_native_id())
        got.append(ps.amplitudes(small.bits, ws=ws, stream=side))

    pw.amplitudes_device(bits, ww, out, stream=busy)
    torch.cuda.synchronize()
    for _ in range(60):  # a few hundred milliseconds of another stream's work
        pw.amplitudes_device(bits, ww, out, stream=busy)
    done.record(busy)
    t = threading.Thread(target=call)
    t.start()
    t.join()
    while os.path.exists(f"/proc/self/task/{tid[0]}"):  # join returns before the thread has let its resources go
        time.sleep(1e-4)
    assert not done.query(), "the end of a thread waited for another stream's work"
    torch.cuda.synchronize()
    assert np.array_equal(got[0], want)


@pytest.mark.parametrize("n,d,nb", [(12, 8, 64), (10, 30, 2)])  # both staged; the narrow kernel and the passes
def test_more_threads_than_staging_blocks(tb, n, d, nb):
    import torch
    c = W.random_circuit(n, d, None, nb, 3)
    plan = tb.Plan.from_circuit(c)
    want = plan.amplitudes(c.bits)
    k = 40
    ws, st = [plan.alloc_workspace(nb) for _ in range(k)], [torch.cuda.Stream() for _ in range(k)]
    torch.cuda.synchronize()
    bad, gate = [], threading.Barrier(k)

    def call(i):
        torch.cuda.set_device(0)
        gate.wait()
        for _ in range(5):
            if not np.array_equal(plan.amplitudes(c.bits, ws=ws[i], stream=st[i]), want):
                bad.append(i)

    ts = [threading.Thread(target=call, args=(i,)) for i in range(k)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
