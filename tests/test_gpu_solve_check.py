"""Kernels of the solve below the C ABI (tests/solve_check.cu, compiled here and run): the
bounded waits of the CG loop's grid barrier and what a wait that gave up leaves behind, and the
range of the product's shares of r^T A r."""
import subprocess

import pytest

from native_check import compile_solve_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return compile_solve_check(tmp_path_factory.mktemp("solve_check"))


def _run(program, what, lines):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.count(": ok") == lines


def test_grid_barrier_gives_up_and_leaves_no_count(program):
    _run(program, "barrier", 9)


def test_shares_of_delta_keep_their_range(program):
    _run(program, "delta", 9)


def test_long_chunks_are_added_in_runs(program):
    _run(program, "runs", 3)
