"""Split grids in 2D: the kernel pair against the fused kernel, which runs where the device has no room for the
pair's U^{m+1/2}: same arithmetic, so the same bits, at the edges of the 32 x 8 tiles, for each exchange mode, limiter
and boundary, and for the pair's compile-time modes (M1, theta = 1) as for the others."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [((3, 3, 1), "full", "minmod", "outflow", {}), ((32, 8, 1), "absorb", "mc", "periodic", {}),
         ((33, 9, 1), "frozen_t", "none", "reflect", {}), ((28, 4, 1), "equilibrium", "mc", "outflow", {}),
         ((61, 23, 1), "full", "none", "reflect", dict(theta_F=0.6, theta_E=0.51)),
         ((64, 16, 1), "absorb", "minmod", "outflow", dict(theta_E=0.75)),
         ((31, 40, 1), "frozen_t", "mc", "periodic", dict(theta_F=0.9, theta_E=0.9)),
         ((97, 7, 1), "full", "mc", "periodic", dict(closure="p1")), ((40, 17, 1), "equilibrium", "minmod", "reflect", {})]


@pytest.mark.parametrize("n,exchange,limiter,bc,kw", CASES)
def test_pair_and_fused_kernel_give_the_same_bits(rhd, monkeypatch, n, exchange, limiter, bc, kw):  # noqa: F811
    case = wl.parity_case("split2d", n, bc=bc, exchange=exchange, limiter=limiter, seed=3, with_v=False, precision="split")
    case["desc"].update(kw)

    def run():
        g = rhd.Grid(case["desc"])
        try:
            g.load_case(case)
            g.set_kernel_timing(True)
            g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
            names = set(g.kernel_times())
            st = g.get_stats()
            out = dict(g.get_moments(), T=g.get_gas_state())
            return names, {k: np.array(v) for k, v in out.items()}, {k: v for k, v in st.items() if k.startswith("n_")}
        finally:
            g.close()

    names, pair, st_pair = run()
    assert names == {"predictor_split_2d", "corrector_split_2d"}
    cells = n[0] * n[1]
    for k in range(60):  # the least device memory that the grid runs in leaves the pair no room
        monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT", str(cells * (60 + 4 * k)))
        try:
            names, fused, st_fused = run()
            break
        except rhd.RhdError as e:
            assert e.status == rhd.ERR_OOM
    else:
        pytest.fail("no limit let the grid run")
    assert names == {"subcycle_fused_split"}
    for k in pair:
        assert np.array_equal(pair[k], fused[k], equal_nan=True), k
    assert st_pair == st_fused
