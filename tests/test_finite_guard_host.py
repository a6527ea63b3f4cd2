"""Planner host check: a plan leaves zeros out only when nothing can turn a zero into
something else (0 x inf is NaN). Compiles tests/host/finite_guard_check.cpp against the
planner sources with the host compiler; no GPU and no device code involved."""
import subprocess

import pytest

from test_tile_skip_host import _compile


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    return _compile(tmp_path_factory, "finite_guard_check")


def _determined(checker, *args):
    r = subprocess.run([checker, *map(str, args)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return int(r.stdout.split("determined=")[1])


PLANS = [(8, 34, 0, 0), (8, 33, 0, 0), (7, 30, 0, 1), (7, 31, 0, 2), (9, 34, 4, 0), (9, 33, 2, 0)]


@pytest.mark.parametrize("plan", PLANS)
def test_ordinary_gates_leave_zeros_out(checker, plan):
    assert _determined(checker, *plan) > 0
    # far from unitary, but within range: row 0, a middle row, the last row
    assert _determined(checker, *plan, 0, 3, "1e3", 3, 5, "1e-3", 7 if plan[0] > 7 else 6, 2, "1e2") > 0


# a gate of row 0, of its first slot, of a middle row, of the last row (an open plan's
# band), of the last slot
@pytest.mark.parametrize("value", ["inf", "nan", "1e39"])  # 1e39 is infinite in FP32
@pytest.mark.parametrize("plan", PLANS)
def test_non_finite_gates_leave_nothing_out(checker, plan, value):
    n, d = plan[:2]
    for q, t in ((0, 0), (0, 4), (0, d), (3, 7), (n - 1, 0), (n - 1, 3), (n - 1, d), (n - 2, d - 1)):
        assert _determined(checker, *plan, q, t, value) == 0, (q, t)


@pytest.mark.parametrize("plan", PLANS)
def test_products_beyond_fp32_leave_nothing_out(checker, plan):
    n = plan[0]
    row0 = [a for t in (1, 2, 3, 4) for a in (0, t, "1e12")]          # one factor of the row-0 boundary
    row = [a for t in (1, 2, 3, 4, 5, 6) for a in (2, t, "1e10")]     # neighbouring steps of one pass
    last = [a for t in (1, 2, 3, 4) for a in (n - 1, t, "1e12")]      # the last row's vectors, the open band
    for args in (row0, row, last):
        assert _determined(checker, *plan, *args) == 0, args


def test_row0_factors_that_only_overflow_together(checker):
    """Each row-0 table is finite in FP32 (address bits 0..11 | 12..): their product is not."""
    assert _determined(checker, 8, 34, 0, 0, 0, 2, "1e30") > 0
    assert _determined(checker, 8, 34, 0, 0, 0, 30, "1e30") > 0
    assert _determined(checker, 8, 34, 0, 0, 0, 2, "1e30", 0, 30, "1e30") == 0
