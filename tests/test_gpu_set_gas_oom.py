"""GPU: a set_gas_state that finds no room for its new arrays.  It leaves the grid as it was, captured subcycle graphs
included, unless it had to give up velocity components that the call drops: then the gas state is not set until the
next call that succeeds."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [((96, 1, 1), "fp64", 4), ((33, 9, 1), "split", 4), ((20, 12, 9), "fp64", 4), ((20, 12, 9), "split", 4)]


def step(g, case):
    g.set_moments(*[case["fields"][k] for k in ("E", "Fx", "Fy", "Fz")])
    g.radiation_subcycle(40, case["chat"], case["dt"])  # more launches than are issued directly: a captured graph
    out = dict(g.get_moments(), T=g.get_gas_state())
    g.get_stats()
    return out


def smallest_grid(rhd, monkeypatch, case, gas):  # noqa: F811
    """A grid with the least device memory that the case runs in, its gas set and stepped."""
    cells = int(np.prod(case["desc"]["n"]))
    for k in range(200):
        monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT", str(cells * (60 + 4 * k) + 1024))
        g = None
        try:
            g = rhd.Grid(case["desc"])
            g.set_gas_state(**gas)
            return g, step(g, case)
        except rhd.RhdError as e:
            if g is not None:
                g.close()
            assert e.status == rhd.ERR_OOM
    pytest.fail("no limit let the grid run")


@pytest.mark.parametrize("n,precision,scale", CASES)
@pytest.mark.parametrize("drops", [False, True])
def test_no_room_for_new_arrays(rhd, monkeypatch, n, precision, scale, drops):  # noqa: F811
    case = wl.parity_case("set_gas_oom", n, bc="outflow", exchange="full", beta_tau=True, seed=11, precision=precision)
    f = case["fields"]
    gas = {k: f[k] for k in ("rho", "T", "vx", "vy", "vz")}
    g, ref = smallest_grid(rhd, monkeypatch, case, gas)
    g.set_gas_state(**gas)
    more = {k: scale * np.ones_like(f["rho"]) for k in ("kP", "kF", "j")}
    other = {k: 2.0 * v for k, v in gas.items() if not (drops and k == "vz")}
    with pytest.raises(rhd.RhdError) as ei:
        g.set_gas_state(**other, **more)
    assert ei.value.status == rhd.ERR_OOM
    if drops:
        with pytest.raises(rhd.RhdError) as ei:
            step(g, case)
        assert ei.value.status == rhd.ERR_STATE
        g.set_gas_state(**gas)
    out = step(g, case)
    g.close()
    for k in ref:
        assert np.array_equal(out[k], ref[k]), k


def test_dropped_velocities_make_room(rhd, monkeypatch):  # noqa: F811
    case = wl.parity_case("set_gas_room", (20, 12, 9), bc="outflow", exchange="full", beta_tau=True, seed=12)
    f = case["fields"]
    g, _ = smallest_grid(rhd, monkeypatch, case, {k: f[k] for k in ("rho", "T", "vx", "vy", "vz")})
    gas = dict(rho=f["rho"], T=f["T"], kP=0.5 * f["rho"], kF=2.0 * f["rho"], j=f["rho"])
    g.set_gas_state(**gas)
    out = step(g, case)
    g.close()
    monkeypatch.delenv("RHD_DEVICE_MEMORY_LIMIT")
    g = rhd.Grid(case["desc"])
    g.set_gas_state(**gas)
    ref = step(g, case)
    g.close()
    for k in ref:
        assert np.max(np.abs(out[k] - ref[k])) <= 1e-12 * case["desc"]["c"] * np.max(np.abs(ref[k])), k


def test_statistics_without_room_for_their_result(rhd, monkeypatch):  # noqa: F811
    """get_stats allocates the partial sums, then the result; where only the first fit, each call says so."""
    case = wl.parity_case("stats_oom", (48, 1, 1), exchange="full", seed=13)
    seen = set()
    for limit in range(3000, 5200, 8):
        monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT", str(limit))
        try:
            g = rhd.Grid(case["desc"])
            g.load_case(case)
        except rhd.RhdError as e:
            assert e.status == rhd.ERR_OOM
            continue
        for _ in range(3):
            try:
                seen.add(np.isfinite(g.get_stats()["sum_E"]))
            except rhd.RhdError as e:
                assert e.status == rhd.ERR_OOM
                seen.add("oom")
        g.close()
    assert seen == {True, "oom"}
