"""Whether the counts per element start a pass at zero is known on the host (csrc/counts_state.h);
captures, replays and passes that were cut short do not mislead it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1006_0532_gb300", "csrc")


def test_no_pass_starts_from_counts_left_over(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "counts_state")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-o", exe, os.path.join(HERE, "counts_state_harness.cpp")],
                   check=True)
    out = dict(line.split() for line in
               subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.splitlines())
    assert out == dict(dirty="0", clears="1")
