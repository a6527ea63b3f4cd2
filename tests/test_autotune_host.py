"""Autotuner cache: a schedule is kept for the circuits it was timed on. How many entries
a pass leaves out as exactly zero depends on the share of monomial gates, so circuits
that differ in it are tuned apart. Host logic only (the timing is replaced)."""
import json

import numpy as np
import pytest

import workloads as W


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    import torch
    from paper_2608_13110_gb300 import autotune, build
    build.build()
    timed = []

    def fake_measure(opts, h, nb, n_rows=8, reps=3, seed=1, monomial=None):
        timed.append(monomial)
        # the default wins on circuits without zeros, a narrow window on the others
        return 1.0 if monomial == 0.0 and not opts["window_bits"] else float(opts["window_bits"] or 99)

    monkeypatch.setattr(autotune, "measure", fake_measure)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "host")
    monkeypatch.setenv("TB_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    return autotune, timed, tmp_path / "tune.json"


def _with_cliffords(n, d, allowed):
    c = W.random_circuit(n, d, None, 4, 1)
    c.cliff = np.random.default_rng(2).choice(np.asarray(allowed, np.uint8), size=c.cliff.shape)
    return c


def _windows(plan):
    return [m for _, m, _ in plan.schedule]


def test_a_dense_circuit_is_not_given_the_schedule_of_one_with_zeros(tuner):
    autotune, timed, _ = tuner
    uniform = autotune.tune(16, nb=4)
    assert uniform["window_bits"] and set(timed) == {None}
    dense = _with_cliffords(12, 32, [k for k in range(24) if k // 4 not in (0, 2)])
    assert _windows(autotune.tuned_plan(dense, nb=4)) == _windows(autotune.Plan.from_circuit(dense))
    assert 0.0 in timed
    diagonal = _with_cliffords(12, 32, [0, 3, 8, 11])
    autotune.tuned_plan(diagonal, nb=4)
    assert 1.0 in timed
    n = len(timed)
    assert autotune.tune(16, nb=4) == uniform and autotune.tune(16, nb=3, monomial=0.3) == uniform
    autotune.tuned_plan(W.random_circuit(12, 32, None, 4, 9), nb=4)  # uniform random Cliffords: a third
    assert len(timed) == n  # served from the cache


def test_entries_timed_without_zeros_are_not_believed(tuner):
    autotune, timed, path = tuner
    old = {"window_bits": 10, "bottom_bits": 10, "top_bits": 10}
    path.write_text(json.dumps({"host|h=16|nb=4": {"opts": old, "ms": 1.0, "tried": 8}}))
    assert autotune.tune(16, nb=4) != old and timed


def test_monomial_cliffords_are_the_matrices_with_two_entries():
    import paper_2608_13110_gb300 as tb
    from paper_2608_13110_gb300 import autotune
    for k in range(24):
        assert (np.count_nonzero(np.abs(tb.clifford_matrix(k)) > 1e-12) == 2) == autotune.MONOMIAL[k]
