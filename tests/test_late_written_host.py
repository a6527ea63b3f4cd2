"""Planner host check: an open plan's late crossings read only rows that the join or the
crossing before them wrote. Compiles tests/host/late_written_check.cpp against the
planner sources with the host compiler; no GPU and no device code involved."""
import subprocess

import pytest

from test_tile_skip_host import _compile


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    return _compile(tmp_path_factory, "late_written_check")


# both parities of d and of the crossing layers (n - k - 1), both joins (k >= 4: tensor
# cores), the narrowest open boundaries; seed 0 is the identity circuit
@pytest.mark.parametrize("n,d,k", [(9, 30, 4), (10, 31, 4), (9, 31, 4), (9, 31, 5), (10, 31, 5), (12, 36, 6), (11, 34, 2),
                                   (10, 33, 1), (11, 33, 1), (9, 25, 6), (10, 25, 6), (9, 26, 3), (12, 37, 8), (11, 37, 8)])
def test_crossings_read_what_was_written(checker, n, d, k):
    for seed in range(6):
        r = subprocess.run([checker, *map(str, (n, d, k, seed))], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout + r.stderr
