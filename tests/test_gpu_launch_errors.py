"""A pass that fails to launch ends the solve with an error, and the solver then still
computes what the oracle does: no graph without that pass is kept.  The failure is made
on the host by the checked build (fh_check_fail_launch) in a child process: inside the
capture of the iterations and (BiCGStab's start) outside it, general two-step,
compile-time two-step and block passes.  Bounds of the other parity tests."""
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
if __name__ == "__main__":
    sys.path.insert(0, os.path.dirname(HERE))
    sys.path.insert(0, HERE)

from parity import Case  # noqa: E402

pytestmark = pytest.mark.gpu

# axes 36 (general two-step), 32 (compile-time two-step), 34 = 2 17 (block passes)
GRIDS = [[2, 36, 36], [2, 32, 32], [2, 34, 34]]
CHUNK = 8


def run_child():
    import paper_1701_04685_gb300 as fh
    from oracle import krylov as OK
    assert fh.checked_build()
    for dims in GRIDS:
        case = Case([[dims[0], 0, 0], [0, dims[1], 0], [0, 0, dims[2]]], {"kind": "dlvp", "alpha": [0.25, 0.2, 0.1]},
                    [(1.0, 0.3), (12.0, 0.2)], np.array([[0.1, -0.05, 0.2]]), np.array([0.3]), nload=1)
        for method in (0, 1):
            if method == 0:
                ref = case.oracle_solve(tol=0.0, max_iter=CHUNK)["E"]
            else:
                ref = np.stack([OK.bicgstab(case.T, case.Gp, case.Cp_o[case.ids], case.C0_o, case.eps0[0], tol=0.0, max_iter=CHUNK)["E"]])
            for nth in (2, 5, 14):
                s = case.product(fh)
                fh.check_fail_launch(nth)
                try:
                    s.solve(case.eps0, tol=0.0, max_iter=CHUNK, method=method, chunk=CHUNK, path=1)
                    raise SystemExit(f"{dims} method {method}: launch {nth} failed and the solve did not")
                except fh.FhError as e:
                    assert e.status == -5, e   # FH_ERR_CUDA
                fh.check_fail_launch(0)
                for _ in range(2):
                    s.solve(case.eps0, tol=0.0, max_iter=CHUNK, method=method, chunk=CHUNK, path=1)
                    assert case.strain_error(s, ref) < (1e-9 if method else 1e-10), (dims, method, nth)
                s.close()
    print("child ok")


def test_failed_launch_ends_the_solve_and_leaves_no_graph():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build(checked=True)
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=dict(os.environ, FH_CHECKED="1"), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


if __name__ == "__main__":
    run_child()
