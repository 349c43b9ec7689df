"""The two-step passes of general lengths (axes of R1 R2 points, 4 <= R1 <= R2 <=
16) against the FP64 oracle: rows and middle columns of every pair of radices'
kind on 2 x L x L grids, axis 0 with the Green step on cubes, and BiCGStab's
operator halves; FP64 within 1e-10 and FP32 within 5e-5 (the bounds of the other
parity tests)."""
import numpy as np
import pytest

from parity import Case, rel

pytestmark = pytest.mark.gpu

LENGTHS = [16, 20, 28, 36, 45, 55, 63, 77, 90, 98, 104, 130, 143, 150, 169, 182, 195, 208, 224, 225, 240]
CUBES = [20, 28, 36, 45]


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


def _case(dims, gen="dlvp", nload=2):
    spec = {"kind": "dlvp", "alpha": [0.25, 0.2, 0.1]} if gen == "dlvp" else {"kind": gen}
    return Case([[dims[0], 0, 0], [0, dims[1], 0], [0, 0, dims[2]]], spec, [(1.0, 0.3), (12.0, 0.2)],
                np.array([[0.1, -0.05, 0.2], [-0.3, 0.3, -0.2]]), np.array([0.25, 0.12]), nload=nload)


def _check(fh, case, n, form=0):
    s = case.product(fh)
    for prec, tol in ((fh.FH_PREC_FP64, 1e-10), (fh.FH_PREC_FP32, 5e-5)):
        out = s.solve(case.eps0, tol=0.0, max_iter=n, precision=prec, form=form)
        ref = case.oracle_solve(tol=0.0, max_iter=n)
        assert case.strain_error(s, ref["E"]) < tol, prec
        assert rel(out["mean_stress"], ref["mean_stress"]) < tol
    # mixed: FP32 iterations, then one in FP64 whose row pass ends after the E update
    s.solve(case.eps0, tol=0.0, max_iter=n, precision=fh.FH_PREC_MIXED)
    ref = case.oracle_solve(tol=0.0, max_iter=n + 1)
    assert case.strain_error(s, ref["E"]) < 5e-5
    s.close()


@pytest.mark.parametrize("L", LENGTHS)
def test_rows_and_columns_match_oracle(fh, L):
    _check(fh, _case([2, L, L], nload=1 if L > 100 else 2), 4)


@pytest.mark.parametrize("n", CUBES)
def test_cubes_match_oracle(fh, n):
    _check(fh, _case([n, n, n], gen="dirichlet", nload=6 if n < 30 else 2), 8)


@pytest.mark.parametrize("dims", [[20, 20, 20], [12, 24, 48]])
def test_bicgstab_matches_oracle(fh, dims):
    from oracle import krylov as OK
    case = _case(dims, nload=2)
    s = case.product(fh)
    kr = np.stack([OK.bicgstab(case.T, case.Gp, case.Cp_o[case.ids], case.C0_o, case.eps0[q], tol=0.0, max_iter=5)["E"]
                   for q in range(2)])
    s.solve(case.eps0, tol=0.0, max_iter=5, method=1)
    assert case.strain_error(s, kr) < 1e-9
    s.close()
