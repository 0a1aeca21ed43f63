"""GPU: the 1D kernel (both precisions) over its plans: runs of up to eight subcycles per launch at sizes one cell
either side of its tiles, with every boundary rule and with the ghost cells refilled between subcycles; one subcycle
per launch where one face alone is periodic; one thread per cell on long lines.  Against the oracle with the bounds of
test_gpu_parity.py, and to the bit against one subcycle per call."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1306_0010_gb300 import workloads as wl
from split_bounds import split_bound
from test_gpu_parity import FP64_TOL, errors, rhd  # noqa: F401

pytestmark = pytest.mark.gpu

DIR = ([[1.2, 0.3, 0.0, 0.0], [0.0] * 4, [0.0] * 4], [[0.8, -0.2, 0.0, 0.0], [0.0] * 4, [0.0] * 4])


def line_case(n, bc, exchange, n_sub, precision, seed=0):
    if not isinstance(bc, str):
        bc = ([bc[0], "outflow", "outflow"], [bc[1], "outflow", "outflow"])
    dirichlet = DIR if "dirichlet" in str(bc) else None
    return wl.parity_case("line", (n, 1, 1), bc=bc, exchange=exchange, beta_tau=True, with_j=n % 2 == 0, n_sub=n_sub,
                          seed=seed, precision=precision, kP_array=n % 3 == 0, dirichlet=dirichlet)


def run(rhd, case, calls):  # noqa: F811
    g = rhd.Grid(case["desc"])
    g.load_case(case)
    for c in calls:
        g.radiation_subcycle(c, case["chat"], case["dt"])
    out = dict(g.get_moments(), T=g.get_gas_state())
    st = {k: v for k, v in g.get_stats().items() if k.startswith("n_") and k != "n_subcycles"}
    g.close()
    return out, st


def check(case, out):
    ref, _ = orc.subcycles(case)
    tol = FP64_TOL if case["desc"]["precision"] == "fp64" else split_bound(case, case["n_sub"])
    assert max(errors(out, ref, case["desc"]).values()) <= tol


@pytest.mark.parametrize("precision", ["fp64", "split"])
@pytest.mark.parametrize("n,bc,exchange,n_sub", [
    (16, "reflect", "full", 17), (15, "periodic", "full", 25), (17, ("reflect", "outflow"), "frozen_t", 17),
    (33, "dirichlet", "full", 25), (31, "reflect", "frozen_t", 25), (47, ("dirichlet", "reflect"), "full", 17),
    (3, "periodic", "full", 17), (3, "reflect", "full", 25), (4, "outflow", "absorb", 17), (64, "periodic", "equilibrium", 17),
    (49, ("outflow", "dirichlet"), "frozen_t", 25), (130, ("outflow", "reflect"), "full", 9),
    (40, ("periodic", "reflect"), "full", 9), (33, ("dirichlet", "periodic"), "full", 9)])
def test_runs_of_subcycles(rhd, n, bc, exchange, n_sub, precision):  # noqa: F811
    case = line_case(n, bc, exchange, n_sub, precision, seed=n)
    out, st = run(rhd, case, [n_sub])
    check(case, out)
    single, st1 = run(rhd, case, [1] * n_sub)
    assert st == st1
    for k in out:
        assert np.array_equal(out[k], single[k]), k


@pytest.mark.parametrize("n,precision", [(8817, "fp64"), (8816, "fp64"), (35265, "split"), (35264, "split"), (4001, "fp64"),
                                         (16001, "split")])
@pytest.mark.parametrize("bc", ["periodic", ("reflect", "outflow")])
def test_long_lines(rhd, n, precision, bc):  # noqa: F811
    """Also piece by piece: 600 cells of a long line as a line of their own (two threads per cell, several subcycles
    per launch) have the same bits beyond the reach of the piece's ends.  (In FP32 the oracle is no measure here:
    among so many random cells some face value sits on the light cone to rounding, and is limited or not.)"""
    case = line_case(n, bc, "full", 5, precision, seed=3)
    out, st = run(rhd, case, [5])
    if precision == "fp64":
        check(case, out)
    single, st1 = run(rhd, case, [2, 1, 2])
    assert st == st1
    for k in out:
        assert np.array_equal(out[k], single[k]), k
    reach = 3 * 5
    for a in (0, n // 2, n - 600):
        piece = dict(case, desc=dict(case["desc"], n=(600, 1, 1)),
                     fields={k: None if v is None else v[:, :, a:a + 600] for k, v in case["fields"].items()})
        part, _ = run(rhd, piece, [5])
        for k in out:
            assert np.array_equal(part[k][:, :, reach:-reach], out[k][:, :, a + reach:a + 600 - reach]), (k, a)


@pytest.mark.parametrize("n,bc", [(40, "reflect"), (9001, "periodic")])
def test_no_alloc_entry_point_is_the_same_kernel(rhd, n, bc):  # noqa: F811
    import torch

    case = line_case(n, bc, "full", 5, "fp64", seed=4)
    ref, _ = run(rhd, case, [5])
    f = {k: torch.tensor(np.ascontiguousarray(v), device="cuda") for k, v in case["fields"].items() if v is not None}
    out = {k: torch.empty_like(f["E"]) for k in ("E", "Fx", "Fy", "Fz", "T")}
    rhd.subcycle_noalloc(case["desc"], 5, case["chat"], case["dt"], *[f[k] for k in ("E", "Fx", "Fy", "Fz", "rho", "T")],
                         *[out[k] for k in ("E", "Fx", "Fy", "Fz", "T")],
                         **{k: f[k] for k in ("vx", "vy", "vz", "kP", "kF", "j") if k in f})
    for k in ref:
        assert np.array_equal(out[k].cpu().numpy().reshape(ref[k].shape), ref[k]), k
