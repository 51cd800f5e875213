"""The FP64 form's elementary functions (csrc/math64.h) on the device, with its own FP32 seeds: none
is less accurate than the library's function that it stands for."""
import os
import subprocess

import pytest

from paper_1006_0532_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_less_accurate_than_the_library(tmp_path):
    exe = str(tmp_path / "math64_device")
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, "-o", exe,
                    os.path.join(HERE, "math64_device.cu")], check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    worst = {k: (float(a), float(b)) for k, a, b in (line.split() for line in lines if line)}
    assert set(worst) == {"log", "cos", "sin", "rcp", "root", "rcbrt", "quotient"}
    for name, (ours, library) in worst.items():
        assert ours <= library, worst
    # rounded once: the correctly rounded result, but for a part in 2^30 of the arguments
    for name in ("rcp", "root", "quotient"):
        assert worst[name][0] <= 0.5001, worst
