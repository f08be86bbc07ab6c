"""The calls go on working, with the same results, after a device reset: what
the library keeps for a kernel holds for one CUDA context only.  The reset
runs in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


def test_calls_after_a_device_reset():
    from paper_2404_01249_gb300 import build
    build.build()
    worker = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_reset_worker.py")
    r = subprocess.run([sys.executable, worker], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout + r.stderr
