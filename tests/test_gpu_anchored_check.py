"""Kernels of the per-anchor forms below the C ABI (tests/anchored_check.cu, compiled here and
run): the precision of the weights' column sums."""
import subprocess

import pytest

from native_check import compile_anchored_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return compile_anchored_check(tmp_path_factory.mktemp("anchored_check"))


def _run(program, what, lines):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.count(": ok") == lines


def test_weight_sums_are_widened_every_32_rows(program):
    _run(program, "weights", 1)
