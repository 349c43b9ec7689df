"""The three variants of the cluster kernel against the FP64 oracle: staged (primes above
13, small unsplit lengths, FP64 lengths of 2, 3 and 5), general (single warps, 7, 11, 13,
large radices), powers of two; both cluster sizes and precisions, two- and three-
dimensional patterns with two axes.  Every grid here fits a cluster in both precisions, and
the solve has to take it.  FP64 within 1e-10, FP32 within 5e-5 (the bounds of the other
parity tests)."""
import numpy as np
import pytest

from parity import Case, rel

pytestmark = pytest.mark.gpu

GRIDS = [[17, 17], [18, 18], [3, 51], [27, 27], [8, 152], [12, 60], [5, 5], [2, 34], [24, 72], [12, 240], [60, 60], [90, 90], [22, 22],
         [26, 52], [16, 224], [10, 210], [33, 33], [96, 96], [32, 64], [1, 17, 34], [1, 20, 60], [1, 14, 28], [1, 8, 24]]


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


@pytest.mark.parametrize("dims", GRIDS, ids=["x".join(map(str, d)) for d in GRIDS])
def test_kinds_match_oracle(fh, dims):
    d = len(dims)
    case = Case(np.diag(dims).tolist(), {"kind": "dlvp", "alpha": [0.25, 0.2, 0.1][:d]}, [(1.0, 0.3), (12.0, 0.2)],
                np.full((1, d), 0.07), np.array([0.3]), nload=2 if d == 2 else 1)
    s = case.product(fh)
    assert len(case.pattern.dims) == 2
    n = 8
    ref = case.oracle_solve(tol=0.0, max_iter=n)
    for prec, tol in ((fh.FH_PREC_FP64, 1e-10), (fh.FH_PREC_FP32, 5e-5)):
        for cluster in (8, 16):
            out = s.solve(case.eps0, tol=0.0, max_iter=n, precision=prec, path=2, cluster=cluster)
            assert out["path"] == 2 and out["cluster"] == cluster
            assert case.strain_error(s, ref["E"]) < tol, (prec, cluster)
            assert rel(out["mean_stress"], ref["mean_stress"]) < tol
    s.close()
