"""GPU: the split kernels' HLL flux at faces without waves is the average of the fluxes, rounded the same way in each
of the functions that form it, and an average of zeros with the M1 closure (hll_average_check.cu)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1306_0010_gb300", "csrc")


def test_average_is_rounded_as_a_sum():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1306_0010_gb300 import build

    os.makedirs(build.BUILD, exist_ok=True)
    exe = os.path.join(build.BUILD, "hll_average_check")
    subprocess.run([build.nvcc(), "-std=c++17", "-O3", *build.ARCH, "-I", CSRC, os.path.join(HERE, "hll_average_check.cu"),
                    "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    assert [int(v) for v in out.split()] == [0, 0, 0, 0], out
