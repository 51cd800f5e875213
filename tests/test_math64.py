"""The FP64 form's elementary functions (csrc/math64.h), compiled for the host."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1006_0532_gb300", "csrc")


def test_errors_in_units_in_the_last_place(tmp_path):
    """Every function within two units in the last place of the exact value (a table entry, a
    series and one or two sums, each rounded once), with the library's behaviour at zero,
    below it and for NaN, where the FP32 seeds do not reach."""
    exe = str(tmp_path / "math64")
    try:
        subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "math64_harness.cpp"),
                        "-o", exe], check=True)
    except FileNotFoundError:
        pytest.skip("no g++")
    out = dict(line.split() for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines())
    assert out.pop("special") == "1"
    assert set(out) == {"log", "cos", "sin", "rcp", "root", "rcbrt"}
    for k, v in out.items():
        assert float(v) < 2.0, (k, v)


def test_widened_is_the_conversion(tmp_path):
    exe = str(tmp_path / "widened")
    try:
        subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "math64_widened_harness.cpp"),
                        "-o", exe], check=True)
    except FileNotFoundError:
        pytest.skip("no g++")
    bad, n = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert bad == "0" and int(n) > 1000000
