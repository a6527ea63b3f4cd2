"""Planner host checks: the tiles that the boundary passes leave out, and the rows
that an open plan's join and late crossings leave out, are exactly zero. Compiles
tests/host/tile_skip_check.cpp and late_skip_check.cpp against the planner sources
with the host compiler; no GPU and no device code involved."""
import os
import subprocess

import pytest

from test_pass_steps_host import CSRC, ROOT, _cuda_include


def _compile(tmp_path_factory, name):
    import shutil
    cxx, inc = shutil.which("g++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp(name) / name)
    srcs = [os.path.join(ROOT, "tests", "host", name + ".cpp")] + [
        os.path.join(CSRC, f) for f in ("plan.cpp", "tc_plan.cpp", "open_plan.cpp")]
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", inc, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                        *srcs, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return exe


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    return _compile(tmp_path_factory, "tile_skip_check")


@pytest.fixture(scope="module")
def late_checker(tmp_path_factory):
    return _compile(tmp_path_factory, "late_skip_check")


# n, d, seed, precision, every odd_gates-th gate dense, window sizes: both
# parities of d, every arithmetic, one or several determined bits per pass, the
# identity circuit (seed 0: every outside bit determined) and dense gates only
@pytest.mark.parametrize("args", [
    (9, 32, 1, 0, 0), (8, 33, 2, 0, 0), (9, 36, 3, 0, 7, 5, 10, 9), (7, 35, 4, 0, 0, 10, 10, 5),
    (8, 32, 5, 0, 0, 5, 9, 8), (6, 36, 0, 0, 0), (6, 31, 0, 0, 0), (7, 30, 6, 1, 0), (6, 33, 7, 1, 0),
    (7, 30, 8, 2, 0), (6, 31, 9, 2, 5), (6, 32, 0, 1, 0), (6, 30, 10, 0, 1), (2, 30, 11, 0, 0), (3, 26, 12, 0, 0),
])
def test_left_out_tiles_are_zero(checker, args):
    r = subprocess.run([checker, *map(str, args)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    frac = float(r.stdout.split("visited=")[1])
    if args[4] == 1:
        assert frac == 1.0  # dense gates: nothing is zero
    elif args[2] == 0:
        assert frac < 0.3   # identity circuit


def test_some_tiles_are_left_out(checker):
    """Random Cliffords fix the parity of neighbouring bits one time in nine."""
    r = subprocess.run([checker, "12", "36", "21", "0", "0"], capture_output=True, text=True)
    assert r.returncode == 0 and float(r.stdout.split("visited=")[1]) < 0.95, r.stdout


# n, d, k, seed: both parities of d and of the crossing layers, the tensor-core
# join (k >= 4) and the FP32 one, the identity circuit (seed 0)
@pytest.mark.parametrize("args", [(9, 30, 4, 1), (10, 31, 4, 2), (9, 31, 5, 3), (12, 36, 6, 4), (11, 34, 2, 5),
                                  (10, 33, 1, 6), (9, 32, 4, 0), (9, 31, 3, 0), (10, 40, 10 - 1, 7)])
def test_left_out_rows_are_zero(late_checker, args):
    r = subprocess.run([late_checker, *map(str, args)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    if args[3] == 0:
        assert float(r.stdout.split("visited=")[1]) < 0.3, r.stdout
