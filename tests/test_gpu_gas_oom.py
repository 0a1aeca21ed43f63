"""GPU: a gas step that finds no room for its arrays at any one of its allocations, and is called again once there is
room (the two-pass kernels' buffers given up for the fused kernel's): the second call has all of them."""
import numpy as np
import pytest

from paper_1306_0010_gb300 import workloads as wl
from test_gpu_gas import rhd  # noqa: F401

pytestmark = pytest.mark.gpu


def test_gas_step_after_no_room(rhd, monkeypatch):  # noqa: F811
    n = (12, 10, 9)
    cells = 12 * 10 * 9
    case = wl.gas_case("gas_oom", n, seed=3, precision="split", with_v=False, beta_tau=False)
    fused = dict(variant="fused", tile=(32, 8), z_chunk=9, staging="cpasync")

    def two_steps(g):
        g.gas_step(case["dt_gas"])
        g.gas_correct()
        return {k: np.array(v) for k, v in g.get_gas().items()}

    g = rhd.Grid(case["desc"])
    g.load_case(case)
    ref = two_steps(g)
    g.close()
    retried = 0
    for k in range(120):
        monkeypatch.setenv("RHD_DEVICE_MEMORY_LIMIT", str(cells * (120 + 2 * k) + 1024))
        try:
            g = rhd.Grid(case["desc"])
        except rhd.RhdError as e:
            assert e.status == rhd.ERR_OOM
            continue
        g.load_case(case)
        out = None
        try:
            out = two_steps(g)
        except rhd.RhdError as e:
            assert e.status == rhd.ERR_OOM
            g.set_launch_config(fused)  # gives back 48 bytes a cell, enough where at most the velocity was missing
            try:
                out = two_steps(g)
                retried += 1
            except rhd.RhdError as e2:
                assert e2.status == rhd.ERR_OOM
        else:
            k = -1
        g.close()
        if out is None:
            continue
        for q in ref:
            assert np.array_equal(out[q], ref[q]), q
        if k < 0:
            break
    else:
        pytest.fail("no limit let the step run")
    assert retried >= 8
