"""GPU: grids of three cells in one or two directions and hundreds in another, and faces of which one alone is
periodic, where the plans choose their extreme tiles, against the oracle with the bounds of test_gpu_parity.py."""
import pytest

from oracle import oracle as orc
from paper_1306_0010_gb300 import workloads as wl
from split_bounds import split_bound
from test_gpu_parity import FP64_TOL, errors, rhd  # noqa: F401

pytestmark = pytest.mark.gpu

HALF = (["periodic", "outflow", "reflect"], ["outflow", "periodic", "periodic"])


@pytest.mark.parametrize("precision", ["fp64", "split"])
@pytest.mark.parametrize("bc", ["periodic", "reflect", HALF], ids=["periodic", "reflect", "half"])
@pytest.mark.parametrize("n", [(3, 300, 1), (300, 3, 1), (3, 3, 200), (3, 200, 3), (200, 3, 3), (8, 32, 5), (33, 7, 4)])
def test_thin_grids(rhd, n, bc, precision):  # noqa: F811
    case = wl.parity_case("thin", n, bc=bc, exchange="full", beta_tau=True, with_j=True, kP_array=n[0] == 3, n_sub=4, fmax=0.5,
                          seed=sum(n), precision=precision)
    g = rhd.Grid(case["desc"])
    g.load_case(case)
    g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
    out = dict(g.get_moments(), T=g.get_gas_state())
    g.get_stats()
    g.close()
    ref, _ = orc.subcycles(case)
    tol = FP64_TOL if precision == "fp64" else split_bound(case, case["n_sub"])
    assert max(errors(out, ref, case["desc"]).values()) <= tol
