"""The sum slots of the solves that run in one launch: no schedule of the blocks lets one read a
sum of another pass (csrc/eulerian_ops.h, pcg_sum_slot, which the kernels index with)."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1006_0532_gb300", "csrc")


def test_no_schedule_mixes_two_passes(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "slots")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, "-o", exe, os.path.join(HERE, "pcg_slots_harness.cpp")],
                   check=True)
    out = dict(line.split() for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines())
    assert out["places"] == "1"
    assert int(out["shared"]) > 0      # the search finds the fault where there is one
    assert out["library"] == "0"


def test_kernels_take_their_slots_from_it():
    src = open(os.path.join(CSRC, "k_eulerian.cu")).read()
    code = re.sub(r"//[^\n]*", "", src)
    # every access to the slots: their base in the arguments, and places by the function
    uses = re.findall(r"[^\n]*a\.slots[^\n]*", code)
    assert uses
    for line in uses:
        assert "pcg_sum_slot" in line or "solve_totals" in line, line
    assert len(re.findall(r"eops::pcg_sum_slot\(pass, which, ", code)) == 3
