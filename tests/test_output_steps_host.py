"""Planner host check: output bits change only the steps whose coefficients the pass
kernels choose per bitstring. Compiles tests/host/output_step_check.cpp against the
planner sources with the host compiler; no GPU and no device code involved."""
import subprocess

import pytest

from test_tile_skip_host import _compile


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    return _compile(tmp_path_factory, "output_step_check")


# n, d, seed, window sizes: both parities of n and d, sweeps that end forward
# and reversed, every window size at the top and at the bottom
@pytest.mark.parametrize("args", [
    (9, 32, 1), (8, 33, 2), (9, 36, 3, 5, 10, 9), (7, 35, 4, 10, 10, 5), (8, 32, 5, 5, 9, 8), (6, 40, 6, 9, 10, 7),
    (9, 41, 7, 6, 10, 7), (3, 30, 8), (8, 44, 9, 9, 10, 7), (3, 27, 10), (12, 56, 11), (11, 61, 12, 9, 8, 6),
])
def test_output_bits_change_only_output_steps(checker, args):
    r = subprocess.run([checker, *map(str, args)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
