"""Host check of the marching gas kernels' index arithmetic (no GPU): gas_march_check.cpp walks every thread of every
CTA through the functions that the kernels call, at the edges of tiles and of chunks of planes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_access_of_a_march_is_in_bounds():
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = [d for d in ("/usr/local/cuda/include", os.path.join(os.environ.get("CUDA_HOME", ""), "include"))
           if os.path.exists(os.path.join(d, "cuda_runtime.h"))]
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    os.makedirs(os.path.join(ROOT, "_build"), exist_ok=True)
    exe = os.path.join(ROOT, "_build", "gas_march_check")
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I",
                        os.path.join(ROOT, "paper_1306_0010_gb300", "csrc"), "-I", inc[0],
                        os.path.join(ROOT, "tests", "gas_march_check.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("ok "), r.stdout
