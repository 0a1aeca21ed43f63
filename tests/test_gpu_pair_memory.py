"""GPU: the memory that the kernel pairs (FP64 in 2D and 3D, split in 2D) and the 1D kernel take beyond a grid's own
arrays is spare.  A context whose device memory holds its arrays and no more runs on the fused kernels, whichever
array comes last: an ensemble's last grid, the velocity, the opacities, the gas step's scratch.  The fused kernels are
held to the oracle with the bounds of test_gpu_parity.py."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1306_0010_gb300 import workloads as wl
from split_bounds import split_bound
from test_gpu_parity import FP64_TOL, errors, rhd  # noqa: F401

pytestmark = pytest.mark.gpu

STATE = {"fp64": 80, "split": 84}  # bytes per cell: E and G twice, T, rho (and its FP32 copy)
ARRAY = {"fp64": 8, "split": 12}   # one more array (and its FP32 copy)
SMALL = 4096                       # statistics, reduction buffers, ensemble tables


def state(g):
    return dict(g.get_moments(), T=g.get_gas_state())


def check(case, out):
    ref, _ = orc.subcycles(case)
    tol = FP64_TOL if case["desc"]["precision"] == "fp64" else split_bound(case, case["n_sub"])
    assert max(errors(out, ref, case["desc"]).values()) <= tol


@pytest.mark.parametrize("n,precision,bc", [((19, 13, 11), "fp64", "outflow"), ((16, 16, 33), "fp64", "periodic"),
                                            ((33, 17, 1), "fp64", "reflect"), ((64, 9, 1), "split", "outflow"),
                                            ((100, 1, 1), "fp64", "periodic"), ((130, 1, 1), "split", "reflect")])
def test_optional_arrays_take_the_pairs_room(rhd, monkeypatch, n, precision, bc):  # noqa: F811
    cells = int(np.prod(n))
    case = wl.parity_case("pair_memory", n, bc=bc, exchange="full", beta_tau=True, with_j=True, kP_array=True, n_sub=6,
                          seed=n[0], precision=precision)
    monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT", str(cells * (STATE[precision] + 6 * ARRAY[precision]) + 512))
    g = rhd.Grid(case["desc"])
    g.load_case(case)
    g.set_kernel_timing(True)
    g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
    assert set(g.kernel_times()) == {"subcycle_fused_" + precision}
    out = state(g)
    g.get_stats()
    g.close()
    check(case, out)


@pytest.mark.parametrize("n,precision", [((9, 8, 7), "fp64"), ((33, 9, 1), "split"), ((20, 11, 1), "fp64")])
def test_gas_step_takes_the_pairs_room(rhd, monkeypatch, n, precision):  # noqa: F811
    cells = int(np.prod(n))
    ext = [k + 4 if k > 1 else 1 for k in n]
    m = int(np.prod(ext))
    faces = sum(m // e * (e + 1) for e, k in zip(ext, n) if k > 1)
    scratch = 8 * (5 * m + 8 * cells + 5 * faces) if precision == "fp64" else 4 * (5 * m + 4 * cells)
    case = wl.gas_case("pair_gas", n, seed=4, precision=precision)

    def run():
        g = rhd.Grid(case["desc"])
        g.load_case(case)
        g.radiation_subcycle(6, case["chat"], case["dt"])  # a captured graph of the kernels of that time
        g.gas_step(case["dt_gas"])
        g.radiation_subcycle(6, case["chat"], case["dt"])
        g.gas_correct()
        out = dict(state(g), **g.get_gas())
        g.get_stats()
        g.close()
        return out

    ref = run()
    monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT", str(cells * (STATE[precision] + 3 * ARRAY[precision]) + scratch + SMALL))
    out = run()
    # FP64: the pair and the fused kernel round differently (each within FP64_TOL of the oracle); split: the same bits
    tol = 2 * FP64_TOL if precision == "fp64" else 0.0
    scale = {"T": np.max(ref["T"]), "rho": np.max(ref["rho"]), "E": np.max(ref["E"])}
    for k in ref:
        s = scale.get(k, case["desc"]["c"] * (scale["E"] if k[0] == "F" else 1.0))
        assert np.max(np.abs(out[k] - ref[k])) <= tol * s, k


@pytest.mark.parametrize("arrays", [False, True])
def test_ensemble_without_room_for_the_pair(rhd, monkeypatch, arrays):  # noqa: F811
    cases = [wl.parity_case("pair_ens", n, bc=bc, exchange="full", beta_tau=arrays, with_j=arrays, kP_array=arrays,
                            n_sub=3, seed=60 + i)
             for i, (n, bc) in enumerate([((12, 9, 7), "outflow"), ((17, 16, 33), "periodic"), ((8, 8, 40), "reflect")])]
    cells = [int(np.prod(c["desc"]["n"])) for c in cases]

    def run():
        e = rhd.Ensemble([c["desc"] for c in cases])
        for i, c in enumerate(cases):
            e.load_case(i, c)
        e.set_kernel_timing(True)
        e.subcycle(3, cases[0]["chat"], [c["dt"] for c in cases])
        names = set(e.kernel_times())
        out = [dict(e.get_moments(i), T=e.get_gas_state(i)) for i in range(len(cases))]
        e.get_stats()
        e.close()
        return names, out

    assert run()[0] == {"ensemble_predictor_fp64", "ensemble_corrector_fp64"}
    monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT",
                       str(sum(cells) * (STATE["fp64"] + (6 * ARRAY["fp64"] if arrays else 0)) + 4 * SMALL))
    names, out = run()
    assert names == {"ensemble_fp64"}
    for c, o in zip(cases, out):
        check(c, o)
