"""Host-side check of the order of calls over streams (csrc/call_order.h) with a fake runtime in the place of CUDA: a
call under another current device, captured streams, and which calls wait for which.  No GPU is used."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1301_1215_gb300", "csrc")


def test_order_of_calls(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "call_order_check")
    subprocess.run([gxx, "-std=c++17", "-Wall", "-I", CSRC, os.path.join(HERE, "host", "call_order_check.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
