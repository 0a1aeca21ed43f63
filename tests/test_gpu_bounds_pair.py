"""GPU: the kernel pairs of 2D grids (split and FP64) and the 1D kernel's runs of several subcycles in the
bounds-checked debug library: no index leaves its array at the edges of their tiles, for any boundary rule, with and
without ghost layers of U^{m+1/2}, and the results match the oracle.  The debug library is loaded in a process of its
own (this file run as a program)."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SIZES = [(3, 3, 1), (32, 8, 1), (33, 9, 1), (31, 17, 1), (97, 5, 1), (16, 33, 1), (3, 1, 1), (17, 1, 1), (129, 1, 1)]
BCS = ["periodic", (["reflect", "periodic", "outflow"], ["outflow", "periodic", "outflow"]),
       (["periodic", "outflow", "outflow"], ["periodic", "reflect", "outflow"]),
       (["dirichlet", "reflect", "outflow"], ["reflect", "dirichlet", "outflow"])]


def test_no_index_out_of_range():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1306_0010_gb300 import build

    build.build()
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    rows = [json.loads(x) for x in r.stdout.splitlines() if x.startswith("{")]
    assert len(rows) == 2 * len(SIZES) * len(BCS)
    for row in rows:
        assert row["checked"] == 1 and row["status"] == 0 and row["violations"] == 0, row
        assert row["error"] <= row["bound"], row


def main():
    sys.path.insert(0, os.path.dirname(HERE))
    from bounds_sweep import D, errors, stats_or_status
    from oracle import oracle as orc
    from paper_1306_0010_gb300 import rhd, workloads as wl
    from split_bounds import split_bound

    rhd.lib(rhd.DEBUG_LIB_PATH)
    for i, n in enumerate(SIZES):
        for b, bc in enumerate(BCS):
            for precision in ("split", "fp64"):
                case = wl.parity_case("bounds", n, bc=bc, exchange="full", beta_tau=True, with_j=b % 2 == 0, n_sub=20,
                                      seed=10 * i + b, precision=precision, kP_array=b > 1,
                                      dirichlet=D["dirichlet"] if b == 3 else None)
                g = rhd.Grid(case["desc"])
                g.load_case(case)
                g.reset_stats()
                g.radiation_subcycle(case["n_sub"], case["chat"], case["dt"])
                st, status, msg = stats_or_status(g.get_stats)
                out = dict(g.get_moments(), T=g.get_gas_state())
                g.close()
                ref, _ = orc.subcycles(case)
                print(json.dumps({"n": n, "bc": b, "precision": precision, "checked": int(rhd.lib().rhd_bounds_checked()),
                                  "status": status, "violations": None if st is None else st["bounds_violations"],
                                  "message": msg, "error": errors(out, ref, case["desc"]),
                                  "bound": 1e-12 if precision == "fp64" else split_bound(case, case["n_sub"])}),
                      flush=True)


if __name__ == "__main__":
    main()
