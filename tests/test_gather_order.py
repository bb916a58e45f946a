"""Host check (no GPU) of the degridding's order of the visibilities, and of
gridding plans with a single tile (tile side = grid side), whose footprints
wrap into the tile they start in."""
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
    exe = str(tmp_path_factory.mktemp("order") / "gather_order_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "gather_order_check.cpp"),
                    os.path.join(CSRC, "gather_plan.cpp"), "-o", exe], check=True)
    return exe


# (grid side L, footprint J, gridding tile T, home tile, visibilities M, seed)
@pytest.mark.parametrize("L,J,T,home,M,seed", [
    (16, 2, 16, 16, 500, 1), (16, 8, 16, 16, 500, 2), (32, 6, 32, 32, 20000, 3), (64, 6, 64, 64, 20000, 4),
    (16, 8, 8, 8, 700, 5), (16, 8, 8, 16, 700, 6),      # two tiles a side, the smallest grid
    (64, 4, 16, 64, 3000, 7),                            # one home tile, sixteen gridding tiles
    (512, 6, 16, 32, 9000, 8), (192, 8, 16, 16, 4000, 9), (64, 6, 64, 64, 1, 10), (64, 6, 64, 64, 0, 11)])
def test_degridding_order_and_walk(checker, L, J, T, home, M, seed):
    r = subprocess.run([checker, str(L), str(J), str(T), str(home), str(M), str(seed)], capture_output=True, text=True,
                       timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
