"""The bounds-check build checks the backward product's writes of the pattern's
values against the row's end, in slices of 32 rows too (tests/_checks_backward_run.py,
a child process: the library a process loads is fixed at its first call)."""
import os
import subprocess
import sys

import pytest

from _gpu import need_gpu

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_values_past_a_rows_end_are_skipped_and_reported():
    need_gpu()
    env = dict(os.environ, PACKSELL_CHECKS="1")
    r = subprocess.run([sys.executable, os.path.join(HERE, "_checks_backward_run.py")], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "checks ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
