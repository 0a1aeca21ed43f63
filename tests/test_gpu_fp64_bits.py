"""GPU: the FP64 path's comparisons by bits give what plain comparisons give (any signs, zeros, infinities,
subnormals; a NaN stops a limited slope), and its square root is within two units in the last place of CUDA's."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1306_0010_gb300", "csrc")


def test_fp64_bit_comparisons_and_square_root():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1306_0010_gb300 import build

    os.makedirs(build.BUILD, exist_ok=True)
    exe = os.path.join(build.BUILD, "fp64_bits_check")
    subprocess.run([build.nvcc(), "-std=c++17", "-O3", *build.ARCH, "-I", CSRC, os.path.join(HERE, "fp64_bits_check.cu"),
                    "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    got = dict(zip(out.split()[0::2], (int(v) for v in out.split()[1::2])))
    assert {k: got[k] for k in ("max0", "min0", "minmod", "reaches1", "sqrt_special")} == dict.fromkeys(
        ("max0", "min0", "minmod", "reaches1", "sqrt_special"), 0), out
    assert got["sqrt_ulp"] <= 2, out
