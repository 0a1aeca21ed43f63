"""GPU: the two-pass split kernels' compile-time modes (M1 closure and speeds, theta = 1; predictor: FULL and
EQUILIBRIUM; corrector: ABSORB and FROZEN_T too) against their general instantiations, to the bit.  The general
corrector runs with TMA staging; the general predictor with ABSORB at k_P = 0, which is EQUILIBRIUM (its factor of E is
exactly 1).  Grids: one tile and less,
ragged tiles, every boundary rule, one plane more than a chunk; optional arrays on and off."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

DIR = ([[1.2, 0.3, 0.0, 0.0], [0.9, 0.0, 0.2, 0.0], [1.1, 0.0, 0.0, 0.4]],
       [[0.8, -0.2, 0.0, 0.0], [1.0, 0.0, 0.0, 0.0], [0.7, 0.0, 0.0, -0.1]])
GRIDS = [((5, 3, 3), "outflow"), ((33, 9, 17), (["reflect", "outflow", "periodic"], ["outflow", "reflect", "periodic"])),
         ((64, 16, 9), (["dirichlet", "outflow", "reflect"], ["outflow", "dirichlet", "outflow"]))]


@pytest.fixture(scope="module")
def rhd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1306_0010_gb300 import build, rhd as binding

    build.build()
    binding.lib()
    return binding


def run(rhd, case, staging="cpasync", **kw):
    desc = dict(case["desc"], **kw)
    g = rhd.Grid(desc)
    g.set_launch_config(dict(variant="twopass", tile=(32, 8), z_chunk=8, staging=staging))
    g.load_case(dict(case, desc=desc))
    g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
    out = g.get_conserved()
    out["T"] = g.get_gas_state()
    st = g.get_stats()
    g.close()
    return out, {k: st[k] for k in st if k.startswith("n_")}


@pytest.mark.parametrize("limiter", ["minmod", "mc", "none"])
@pytest.mark.parametrize("exchange", ["full", "equilibrium", "absorb", "frozen_t"])
@pytest.mark.parametrize("i", range(len(GRIDS)))
def test_common_modes_are_the_general_ones(rhd, i, exchange, limiter):
    n, bc = GRIDS[i]
    case = wl.parity_case("modes", n, bc=bc, exchange=exchange, limiter=limiter, beta_tau=True, n_sub=3, seed=600 + i,
                          precision="split", with_j=i != 1, kP_array=i == 2, dirichlet=DIR)
    ref, st_ref = run(rhd, case, staging="tma")
    out, st = run(rhd, case)
    assert st == st_ref
    for k in ref:
        assert np.array_equal(out[k], ref[k]), k
    if exchange == "equilibrium" and case["fields"]["kP"] is None:
        out, st = run(rhd, case, exchange="absorb", kappa_P=0.0)
        assert st == st_ref
        for k in ref:
            assert np.array_equal(out[k], ref[k]), k
