"""GPU: a Marshak run on 2D and 3D grids, whose kernel pairs read the boundary states from device memory (the low x
ghost cells of U^{m+1/2} among them), against the oracle with the bounds of test_gpu_marshak.py."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from split_bounds import split_bound
from test_gpu_marshak import N_QUAD, oracle_run, rhd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,precision", [((48, 5, 1), "fp64"), ((48, 5, 1), "split"), ((40, 4, 3), "fp64"), ((33, 9, 1), "split")])
def test_marshak_on_wider_grids(rhd, n, precision):  # noqa: F811
    case = wl.marshak_case(n[0], precision=precision)
    d = case["desc"]
    for side in ("bc_lo", "bc_hi"):
        d[side] = [d[side][0], "periodic", "periodic"]
    d["n"], d["dx"] = n, (d["dx"][0],) * 3
    case["fields"] = {k: None if v is None else np.ascontiguousarray(np.broadcast_to(v, (n[2], n[1], n[0])))
                      for k, v in case["fields"].items()}
    case["dt"] *= 0.5
    n_sub = 60
    ref = oracle_run(case, n_sub)
    g = rhd.Grid(d)
    g.load_case(case)
    g.marshak_advance(25, case["chat"], case["dt"], 0.0, case["marshak"], n_quad=N_QUAD)
    g.marshak_advance(35, case["chat"], case["dt"], 25 * case["dt"], case["marshak"], n_quad=N_QUAD)
    out = dict(g.get_moments(), T=g.get_gas_state())
    assert g.get_stats()["n_nonfinite"] == 0
    g.close()
    tol = 1e-12 if precision == "fp64" else split_bound(case, n_sub)
    sE = float(np.max(ref["E"]))
    for k, s in (("E", sE), ("Fx", d["c"] * sE), ("T", float(np.max(ref["T"])))):
        assert float(np.max(np.abs(out[k] - ref[k]))) <= tol * s, k
    assert sE > 0.1
