"""GPU: the tuner's candidates include what an untuned grid runs, a configuration that was read from a grid can be put
back, and a 1D grid's tuned time is that of the launches it makes."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu

KEYS = ("variant", "tile", "z_chunk", "staging")


def grid(rhd, n, precision, **kw):  # noqa: F811
    case = wl.parity_case("plan", n, bc="outflow", exchange="full", n_sub=3, seed=5, precision=precision)
    g = rhd.Grid(dict(case["desc"], **kw))
    g.load_case(case)
    return g, case


def conf(c):
    return tuple(c[k] for k in KEYS)


@pytest.mark.parametrize("n,precision,kw", [((40, 40, 40), "split", {}), ((97, 61, 45), "split", {}),
                                            ((40, 40, 40), "split", dict(z_chunk=7)), ((33, 9, 1), "split", {}),
                                            ((40, 40, 40), "fp64", {}), ((40, 40, 40), "fp64", dict(z_chunk=7))])
def test_untuned_configuration_is_a_candidate(rhd, n, precision, kw):  # noqa: F811
    g, case = grid(rhd, n, precision, **kw)
    before = g.launch_config()
    chosen, table = g.autotune(case["chat"], case["dt"], reps=2)
    best = min(c["ms_per_subcycle"] for c in table)
    if precision == "split":
        assert conf(before) in [conf(c) for c in table]
        assert chosen["ms_per_subcycle"] == best
    else:
        assert chosen["ms_per_subcycle"] <= best
    g.set_launch_config(before)
    assert conf(g.launch_config()) == conf(before)
    g.close()


@pytest.mark.parametrize("n,precision", [((40, 40, 40), "split"), ((24, 16, 40), "fp64"), ((33, 9, 1), "fp64")])
def test_read_and_put_back_gives_the_same_steps(rhd, n, precision):  # noqa: F811
    outs = []
    for back in (False, True):
        g, case = grid(rhd, n, precision)
        if back:
            own = g.launch_config()
            g.set_launch_config(dict(own, z_chunk=max(1, own["z_chunk"] - 1)))
            g.set_launch_config(own)
            assert conf(g.launch_config()) == conf(own)
        g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
        outs.append(dict(g.get_moments(), T=g.get_gas_state()))
        g.close()
    for k in outs[0]:
        assert np.array_equal(outs[0][k], outs[1][k]), k


def test_split_ensemble_plan_is_a_candidate(rhd):  # noqa: F811
    cases = [wl.parity_case("plan_ens", n, bc="outflow", exchange="full", n_sub=2, seed=6, precision="split")
             for n in ((20, 12, 10), (33, 9, 17))]
    ens = rhd.Ensemble([c["desc"] for c in cases])
    for i, c in enumerate(cases):
        ens.load_case(i, c)
    before = ens.launch_config()
    chosen, table = ens.autotune(1.0, [c["dt"] for c in cases], reps=2)
    ens.close()
    assert (before["variant"], before["z_chunk"]) in [(c["variant"], c["z_chunk"]) for c in table]
    assert chosen["ms_per_subcycle"] == min(c["ms_per_subcycle"] for c in table)


@pytest.mark.parametrize("precision", ["fp64", "split"])
def test_tuned_time_of_a_1d_grid(rhd, precision):  # noqa: F811
    g, case = grid(rhd, (512, 1, 1), precision)
    T = np.array(g.get_gas_state())
    chosen, _ = g.autotune(case["chat"], case["dt"], reps=50)
    assert np.array_equal(g.get_gas_state(), T)
    g.set_kernel_timing(True)
    g.radiation_subcycle(160, case["chat"], case["dt"])
    (kt,) = g.kernel_times().values()
    g.close()
    assert kt["launches"] < 160  # several subcycles a launch
    # one launch of one subcycle takes 1.7 times as long per subcycle
    assert chosen["ms_per_subcycle"] <= 1.3 * kt["total_ms"] / 160
