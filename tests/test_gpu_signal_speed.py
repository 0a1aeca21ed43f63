"""max_signal_speed, whose kernel passes over the cells that FP32 can tell from the maximum, against NumPy in FP64
on fields where it cannot tell them (equal cells, cells a few FP64 ulps apart), where FP32 under- or overflows, and
on plain random ones.  Tolerance: the value is some ten FP64 operations under a square root; 4e-15 is 18 ulps."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["random", "uniform", "ulps", "ramp", "tiny", "huge", "rest", "nan"])
@pytest.mark.parametrize("n", [(3, 1, 1), (61, 7, 5), (130, 65, 67)])
def test_signal_speed_is_the_fp64_maximum(rhd, kind, n):  # noqa: F811
    case = wl.gas_case("signal", n, seed=5, kF_array=kind == "random", with_v=kind != "rest")
    d, f = case["desc"], {k: (None if v is None else np.array(v)) for k, v in case["fields"].items()}
    g = np.random.default_rng(7)
    if kind not in ("random", "rest"):
        for k in ("rho", "T", "vx", "vy", "vz", "E"):
            f[k] = np.full_like(f["rho"], {"rho": 1.25, "T": 0.75, "E": 2.0}.get(k, 0.125))
    if kind == "ulps":
        f["T"] = f["T"] * (1 + 2.0 ** -52 * g.integers(0, 9, f["T"].shape))
    if kind == "ramp":
        f["T"] = f["T"] * (1 + 1e-7 * np.arange(f["T"].size).reshape(f["T"].shape) / f["T"].size)
    if kind in ("tiny", "huge"):
        s = 1e-33 if kind == "tiny" else 1e30
        f["rho"] = s * (1 + g.random(f["rho"].shape))
        f["T"] = (1e-9 if kind == "tiny" else 1e12) * (1 + g.random(f["T"].shape))
        f["E"] = np.full_like(f["E"], 1e-36)
    if kind == "nan":
        f["T"].flat[-1] = np.nan
    grid = rhd.Grid(dict(d, kappa_rho_pow=0) if kind in ("tiny", "huge") else d)
    grid.load_case(dict(case, fields=f))
    got = grid.max_signal_speed() if kind != "nan" else None
    if kind == "nan":
        with pytest.raises(rhd.RhdError):
            grid.max_signal_speed()
        grid.close()
        return
    grid.close()
    pw = 0 if kind in ("tiny", "huge") else d["kappa_rho_pow"]
    k = f["kF"] if f.get("kF") is not None else d["kappa_F"] * f["rho"] ** pw
    dx = min(d["dx"][a] for a in range(3) if n[a] > 1)
    v2 = 0.0 if f["vx"] is None else f["vx"] ** 2 + f["vy"] ** 2 + f["vz"] ** 2
    q = d["gamma"] * f["rho"] * f["T"] / d["mu_over_kB"] + 4.0 / 9.0 * f["E"] * -np.expm1(-k * dx)
    ref = float(np.max(np.sqrt(v2) + np.sqrt(q / f["rho"])))
    assert abs(got - ref) <= 4e-15 * ref
