"""The library's host code against a stand-in CUDA runtime (CPU only): see
tests/host_calls.py for each check."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("check", ["stream_order", "another_gpu", "other_device"])
def test_host_calls(check):
    r = subprocess.run([sys.executable, os.path.join(HERE, "host_calls.py"), check], capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
