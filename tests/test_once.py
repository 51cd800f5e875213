"""Work done once per device (csrc/once.h) is done before any thread goes on without it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1006_0532_gb300", "csrc")


def test_a_device_counts_as_done_only_after_its_setting(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "once")
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-I", CSRC, "-o", exe, os.path.join(HERE, "once_harness.cpp")],
                   check=True)
    out = dict(line.split() for line in
               subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.splitlines())
    assert out == dict(ready="1", again="0", failure="1", unknown="4")
