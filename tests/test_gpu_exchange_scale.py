"""GPU: the FP64 path has no range of its own.  A case scaled by s in rho, E, F, a_R and E_floor (and kappa by 1/s, so
that every k and the optical depths stay) has the same solution scaled by s; s takes the gas and radiation energy
densities far below and above the FP32 range, which the FP64 exchange's first steps use.  Against the oracle of the
scaled case, with the FP64 path's bound (test_gpu_parity.py)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1306_0010_gb300 import workloads as wl
from test_gpu_parity import FP64_TOL, errors, rhd  # noqa: F401

pytestmark = pytest.mark.gpu

SCALES = [1e-44, 1e-40, 1e-38, 1e-36, 1e-34, 1e-31, 1e-30, 1e-28, 1e-25, 1e-20, 1e20, 1e26, 1e30, 1e36, 1e40]


def scaled(n, s, theta, seed):
    case = wl.parity_case("scale", n, bc="outflow", exchange="full", beta_tau=True, theta=theta, n_sub=3, seed=seed)
    d = case["desc"]
    for k in ("a_rad", "E_floor"):
        d[k] = d[k] * s
    for k in ("kappa_P", "kappa_F"):
        d[k] = d[k] / s
    for k in ("rho", "E", "Fx", "Fy", "Fz"):
        case["fields"][k] = case["fields"][k] * s
    return case


def run(rhd, case):  # noqa: F811
    g = rhd.Grid(case["desc"])
    g.load_case(case)
    g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
    out = dict(g.get_moments(), T=g.get_gas_state())
    g.get_stats()
    g.close()
    return out


@pytest.mark.parametrize("s", SCALES)
@pytest.mark.parametrize("n,theta", [((12, 9, 7), 1.0), ((17, 9, 1), 1.0), ((10, 9, 5), 0.55), ((33, 1, 1), 1.0)])
def test_scaled_case_matches_the_oracle(rhd, n, theta, s):  # noqa: F811
    case = scaled(n, s, theta, seed=len(n))
    ref, _ = orc.subcycles(case)
    e = errors(run(rhd, case), ref, case["desc"])
    assert max(e.values()) <= FP64_TOL, e


@pytest.mark.parametrize("s", [1e-38, 1e-31, 1e30])
def test_scaled_ensemble_matches_the_oracle(rhd, s):  # noqa: F811
    cases = [scaled(n, s, 1.0, 40 + i) for i, n in enumerate([(12, 9, 7), (5, 8, 17)])]
    ens = rhd.Ensemble([c["desc"] for c in cases])
    for i, c in enumerate(cases):
        ens.load_case(i, c)
    ens.subcycle(3, cases[0]["chat"], [c["dt"] for c in cases])
    for i, c in enumerate(cases):
        ref, _ = orc.subcycles(c)
        out = dict(ens.get_moments(i), T=ens.get_gas_state(i))
        assert max(errors(out, ref, c["desc"]).values()) <= FP64_TOL, i
    ens.close()
