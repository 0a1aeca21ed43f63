"""max_signal_speed where FP32 does not see what FP64 sees: a NaN opacity in a slow cell is reported, and cells whose
rho T or k_F lie below the FP32 range are ranked by their FP64 values (tolerance: test_gpu_signal_speed.py)."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = [(61, 7, 5), (130, 65, 67)]


def grid(rhd, n, desc, **fields):  # noqa: F811
    case = wl.gas_case("signal", n, seed=8, kF_array=True, with_v=False)
    f = {k: (None if v is None else np.array(v)) for k, v in case["fields"].items()}
    f.update(fields)
    g = rhd.Grid(dict(case["desc"], **desc))
    g.load_case(dict(case, fields=f))
    return g


def shaped(n, v):
    return np.full((n[2], n[1], n[0]), v)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("bad", [np.nan, -np.nan])
def test_nan_opacity_is_reported(rhd, n, bad):  # noqa: F811
    T, kF = shaped(n, 1.0), shaped(n, 100.0)
    T[-1, -1, -1], kF[-1, -1, -1] = 1e-3, bad
    g = grid(rhd, n, {}, rho=shaped(n, 1.0), T=T, E=1e-3 * T, kF=kF)
    with pytest.raises(rhd.RhdError) as ei:
        g.max_signal_speed()
    assert ei.value.status == rhd.ERR_NONFINITE
    g.close()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("what", ["pressure", "opacity"])
def test_values_below_the_fp32_range(rhd, n, what):  # noqa: F811
    r = np.random.default_rng(9)
    rnd = 1.0 + r.random((n[2], n[1], n[0]))
    if what == "pressure":  # P = rho T / mu ~ 1e-21 from rho T ~ 1e-41
        d = dict(mu_over_kB=1e-20)
        f = dict(rho=shaped(n, 1e-28), T=1e-13 * rnd, E=shaped(n, 1e-35), kF=shaped(n, 1.0))
    else:  # (4/9) E k_F dx ~ 1e-17 from k_F ~ 1e-41, beside P ~ 1e-22
        d = dict(dx=(1e24, 1e24, 1e24))
        f = dict(rho=shaped(n, 1e-22), T=shaped(n, 1.0), E=shaped(n, 1.0), kF=1e-41 * rnd)
    g = grid(rhd, n, d, **f)
    got = g.max_signal_speed()
    g.close()
    base = wl.gas_case("signal", n, seed=8)["desc"]
    mu, gamma = d.get("mu_over_kB", base["mu_over_kB"]), base["gamma"]
    dx = min(d.get("dx", base["dx"]))
    q = gamma * f["rho"] * f["T"] / mu + 4.0 / 9.0 * f["E"] * -np.expm1(-f["kF"] * dx)
    ref = float(np.max(np.sqrt(q / f["rho"])))
    assert abs(got - ref) <= 4e-15 * ref
