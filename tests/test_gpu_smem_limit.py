"""GPU: a launch site remembers the shared-memory limit of all its kernels (smem_limit_check.cu)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1306_0010_gb300", "csrc")


def test_every_kernel_of_a_site_is_remembered():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1306_0010_gb300 import build

    os.makedirs(build.BUILD, exist_ok=True)
    exe = os.path.join(build.BUILD, "smem_limit_check")
    subprocess.run([build.nvcc(), "-std=c++17", "-O1", *build.ARCH, "-I", CSRC, os.path.join(HERE, "smem_limit_check.cu"),
                    "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    assert [int(v) for v in out.split()] == [20, 20, 20], out
