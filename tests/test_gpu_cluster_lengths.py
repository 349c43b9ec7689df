"""The cluster kernel's line transforms by length against the FP64 oracle: one
line per lane (N <= 16), two steps in one warp (N = R1 R2), whole-CTA stages of
large radices (768, primes above 13, 25 * 16), powers of two, and the FP64
schedules on both sides of two points a thread; clusters of 8 and 16, one and
three loads.  FP64 within 1e-10 and FP32 within 5e-5 (the bounds of the other
parity tests)."""
import numpy as np
import pytest

from parity import Case, rel

pytestmark = pytest.mark.gpu

GRIDS = [[2, 4], [3, 9], [7, 14], [13, 26], [16, 16], [6, 30], [15, 45], [24, 24], [4, 512], [96, 96], [60, 180], [17, 34], [8, 768],
         [5, 255], [10, 400], [32, 32], [48, 96], [64, 64]]


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


@pytest.mark.parametrize("cluster", [8, 16])
@pytest.mark.parametrize("dims", GRIDS, ids=["x".join(map(str, d)) for d in GRIDS])
def test_cluster_lines_match_oracle(fh, dims, cluster):
    nload = 3 if dims[0] % 2 else 1
    case = Case([[dims[0], 0], [0, dims[1]]], {"kind": "dlvp", "alpha": [0.25, 0.2]}, [(1.0, 0.3), (12.0, 0.2)],
                np.array([[0.1, -0.05]]), np.array([0.25]), nload=nload)
    s = case.product(fh)
    assert len(case.pattern.dims) == 2
    n = 8
    ref = case.oracle_solve(tol=0.0, max_iter=n)
    for prec, tol in ((fh.FH_PREC_FP64, 1e-10), (fh.FH_PREC_FP32, 5e-5)):
        try:
            out = s.solve(case.eps0, tol=0.0, max_iter=n, precision=prec, path=2, cluster=cluster)
        except fh.FhError as e:
            assert e.status == -8   # the fields do not fit in a cluster of this size
            continue
        assert out["path"] == 2
        assert case.strain_error(s, ref["E"]) < tol, prec
        assert rel(out["mean_stress"], ref["mean_stress"]) < tol
    s.close()
