"""Host test of the split two-pass kernels' planes per CTA (csrc/march_plan.h): the plans whose times its comment states,
and plans within the grid for any size (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# nx, ny, nz, ghost layers -> planes per CTA of the predictor and the corrector
PLANS = {(97, 61, 45, 2): (5, 5), (64, 64, 64, 2): (5, 4), (256, 256, 256, 2): (130, 20), (512, 512, 512, 2): (65, 57),
         (64, 64, 64, 0): (2, 4), (40, 40, 40, 0): (3, 3), (300, 250, 200, 0): (20, 20), (512, 512, 512, 0): (64, 57)}


@pytest.fixture(scope="module")
def plan_exe():
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    os.makedirs(os.path.join(ROOT, "_build"), exist_ok=True)
    exe = os.path.join(ROOT, "_build", "march_plan_check")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1306_0010_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "march_plan_check.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def test_plans_of_known_grids(plan_exe):
    lines = "\n".join(" ".join(map(str, k)) for k in PLANS)
    out = subprocess.run([plan_exe], input=lines, capture_output=True, text=True, check=True).stdout
    assert [tuple(map(int, x.split())) for x in out.splitlines()] == list(PLANS.values())


def test_every_plan_lies_within_the_grid(plan_exe):
    out = subprocess.run([plan_exe, "sweep"], capture_output=True, text=True, check=True, timeout=300).stdout
    bad, n = map(int, out.split())
    assert bad == 0 and n > 10000
