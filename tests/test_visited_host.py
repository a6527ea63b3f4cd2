"""The plan's count of the entries its passes move and of the multiply-adds they execute:
against every visited tile and warp (tests/host/visited_check.cpp, host compiler, no GPU),
and through the API where nothing is zero."""
import subprocess

import pytest

import workloads as W
from test_tile_skip_host import _compile


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    return _compile(tmp_path_factory, "visited_check")


# n, d, seed, window sizes: 8- and 9-bit windows above bit 0 idle warps
@pytest.mark.parametrize("args", [(12, 36, 1), (12, 35, 2), (10, 44, 3, 9, 10, 7), (10, 44, 4, 8, 9, 8), (9, 32, 5),
                                  (9, 42, 6, 8, 8, 9), (8, 28, 7, 10, 10, 5)])
def test_counts_what_the_passes_do(checker, args):
    r = subprocess.run([checker, *map(str, args)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_api_counts():
    import paper_2608_13110_gb300 as tb
    from paper_2608_13110_gb300 import build
    build.build()
    n, d, h = 8, 36, 18
    u = W.random_unitaries(n, d, 1)
    dense = tb.Plan(n, d, extra=[(q, t, u[t, q]) for t in range(d + 1) for q in range(n)])
    assert dense.visited == (dense.info["n_passes"] * 2.0 ** h, dense.info["pass_madds"] * 2.0 ** h)
    e, m = tb.Plan.from_circuit(W.random_circuit(n, d, None, 1, 1)).visited
    assert 0 < e < dense.visited[0] and 0 < m < dense.visited[1]
    assert tb.Plan(n, 24).visited == (0.0, 0.0)  # narrow: no passes
    tc = tb.Plan(n, d, precision="tf32x3", extra=[(q, t, u[t, q]) for t in range(d + 1) for q in range(n)])
    assert tc.visited == (tc.info["n_passes"] * 2.0 ** h, 0.0)
