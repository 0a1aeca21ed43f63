"""GPU: F / c of the moments that a caller hands over is the correctly rounded quotient (div_by_check.cu)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1306_0010_gb300", "csrc")


def test_division_by_the_speed_of_light_is_exact():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1306_0010_gb300 import build

    os.makedirs(build.BUILD, exist_ok=True)
    exe = os.path.join(build.BUILD, "div_by_check")
    subprocess.run([build.nvcc(), "-std=c++17", "-O2", *build.ARCH, "-I", CSRC, os.path.join(HERE, "div_by_check.cu"),
                    "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    n_half, bad_half, n_other, bad_other, bad_p = (int(v) for v in out.split())
    assert n_half > 500000 and n_other > 1 << 20
    assert (bad_half, bad_other, bad_p) == (0, 0, 0), out
