"""Checked build: the record of a failed index check is reported once.  The self test fails
a check in every compiled unit at once; the solves that follow, on kernels of every unit,
are clean (child process, FH_CHECKED=1)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_child():
    import paper_1701_04685_gb300 as fh
    assert fh.checked_build()
    rc, msg = fh.check_selftest()
    assert rc == fh.FH_ERR_INTERNAL and "self test" in msg, (rc, msg)
    for M, path in (([[16, 0], [0, 16]], 2), ([[12, 0], [0, 12]], 2), ([[20, 0], [0, 20]], 1)):
        s = fh.Solver(fh.Pattern(M), fh.generator("dirichlet"), 1)
        s.set_stiffness_phases(np.arange(s.m, dtype=np.uint8) % 2, np.stack([fh.isotropic_stiffness(*fh.lame(E, 0.3), 2) for E in (1.0, 5.0)]))
        s.set_reference(None)
        for prec in (0, 1):
            s.solve(np.eye(3)[:1], tol=0.0, max_iter=2, precision=prec, path=path)
        s.close()
    print("child ok")


def test_records_are_reported_once():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build(checked=True)
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=dict(os.environ, FH_CHECKED="1"), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0 and "child ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


if __name__ == "__main__":
    sys.path.insert(0, ROOT)
    run_child()
