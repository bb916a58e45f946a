"""Host check (no GPU) of the tap weights that the stored G^T G stencils are
built from: they hold the kernels (§5) to FP64 rounding."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1307_4370_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("taps") / "kernel_taps_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "kernel_taps_check.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("kernel", [0, 1])  # Kaiser-Bessel, Gaussian
@pytest.mark.parametrize("J", [2, 4, 6, 8])
def test_tap_weights(checker, J, kernel):
    r = subprocess.run([checker, str(J), str(kernel)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
