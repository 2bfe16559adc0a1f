"""The suites of the grouped deposit, the fused 2D updates and the sort's work
items under the index-checked build (needs a GB300), beside the parity suites
of test_checked_gpu.py: no index leaves its buffer with full items and groups,
ragged strips, shuffled input or drifted particles."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_deposit_field_and_sort_suites_under_the_checked_build():
    from paper_1503_02464_gb300 import build
    build.build(checked=True)
    env = dict(os.environ, PIC_LIBRARY="checked")
    suites = ["tests/test_push_groups_gpu.py", "tests/test_full_items_gpu.py", "tests/test_exact_sums_gpu.py",
              "tests/test_field_step_gpu.py", "tests/test_tape_copy_gpu.py", "tests/test_early_sort_gpu.py",
              "tests/test_sort_gpu.py", "tests/test_adjoint_transpose_gpu.py"]
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider"] + suites,
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert " passed" in r.stdout
