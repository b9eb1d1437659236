"""What is done once per GPU: no call loads device code, since cache creation has
loaded every kernel, and figures of a GPU are kept for that GPU."""
import os
import subprocess
import sys

import pytest

from tests import _native

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_call_waits_for_a_kernel_that_runs_elsewhere():
    _native.helper()  # built before the process below needs it
    for _ in range(2):  # once more if this machine paused the process
        r = subprocess.run([sys.executable, "-m", "tests._code_loading"], cwd=ROOT,
                           stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, timeout=300)
        assert r.returncode == 0, r.stdout
        last = r.stdout.strip().splitlines()[-1]
        if last == "routes 30, late: none":
            return
    raise AssertionError(last)


def test_a_figure_is_kept_once_it_is_known():
    assert _native.helper().helper_per_device() == 55
