"""The gas step's marching kernels (split grids; FP64 grids in 1D) at the edges of their tiles (32 x 8 cells in
2D and 3D, 96 cells in 1D, two ghost layers more in the predictor) and of their chunks of planes, against the
oracle with the bounds of test_gpu_gas.py (derived there)."""
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd, test_gas_step_and_correction_match_oracle as check  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [((28, 4, 9), "split", "periodic", "minmod"), ((29, 5, 17), "split", "reflect", "mc"),
         ((32, 8, 8), "split", "outflow", "none"), ((33, 9, 3), "split", "periodic", "mc"),
         ((64, 16, 1), "split", "reflect", "minmod"), ((61, 13, 1), "split", "outflow", "mc"),
         ((92, 1, 1), "split", "periodic", "minmod"), ((97, 1, 1), "fp64", "reflect", "mc"),
         ((92, 1, 1), "fp64", "outflow", "minmod"), ((193, 1, 1), "fp64", "periodic", "none"),
         ((40000, 1, 1), "fp64", "reflect", "minmod"), ((40001, 1, 1), "split", "outflow", "minmod")]


@pytest.mark.parametrize("n,precision,bc,limiter", CASES)
def test_gas_step_at_tile_edges(rhd, n, precision, bc, limiter):  # noqa: F811
    check(rhd, dict(name="tiles", n=n, precision=precision, bc=bc, limiter=limiter, kF_array=n[0] % 2 == 0))
