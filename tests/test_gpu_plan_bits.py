"""GPU: how a grid is cut into tiles and chunks of planes does not show in its results.  The plan made at creation
(z_chunk = 0: the two kernels' chunks differ) against one chunk length for both, to the bit."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["split", "fp64"])
@pytest.mark.parametrize("n,bc", [((40, 40, 40), "periodic"), ((97, 61, 45), "outflow"), ((70, 33, 9), "reflect"),
                                  ((33, 9, 150), (["outflow", "periodic", "reflect"], ["reflect", "periodic", "outflow"])),
                                  ((130, 120, 70), "outflow")])
def test_planned_chunks_give_the_same_bits(rhd, n, bc, precision):  # noqa: F811
    case = wl.parity_case("plan_bits", n, bc=bc, exchange="full", beta_tau=True, with_j=True, kP_array=n[0] % 2 == 0,
                          n_sub=3, seed=n[2], precision=precision)

    def run(z):
        g = rhd.Grid(dict(case["desc"], z_chunk=z))
        g.load_case(case)
        g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
        out = dict(g.get_moments(), T=g.get_gas_state())
        st = {k: v for k, v in g.get_stats().items() if k.startswith("n_")}
        g.close()
        return out, st

    ref, st_ref = run(0)
    for z in (1, 7, 32, n[2]):
        out, st = run(z)
        assert st == st_ref, z
        for k in ref:
            assert np.array_equal(out[k], ref[k]), (z, k)
