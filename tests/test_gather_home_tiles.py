"""Host check (no GPU) of gridding plans whose visibility sort keeps larger
tiles than the gridding: the sort, hence the order of exported states and of
the bf16 blocks, follows home_T, everything of the gather follows T."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1307_4370_gb300", "csrc")


@pytest.mark.parametrize("L,J,T,home,M,seed", [(512, 6, 16, 32, 6000, 1), (512, 8, 16, 32, 3000, 2),
                                               (128, 2, 8, 32, 2000, 3), (64, 4, 16, 16, 500, 4),
                                               (64, 4, 16, 32, 1, 5), (64, 6, 16, 32, 0, 6)])
def test_home_tiles(tmp_path, L, J, T, home, M, seed):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "gather_home_check")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "gather_home_check.cpp"),
                    os.path.join(CSRC, "gather_plan.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe, str(L), str(J), str(T), str(home), str(M), str(seed)], capture_output=True, text=True,
                       timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
