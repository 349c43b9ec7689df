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


# 2-D patterns on the passes: every radix above 16, one and three loads (an odd
# number of real lines per block), sheared M
PLANES = [[[16, 0], [0, 512]], [[20, 0], [0, 360]], [[24, 0], [0, 480]], [[18, 6], [0, 45]], [[32, 0], [0, 1024]], [[100, 0], [0, 100]],
          [[36, 9], [0, 40]], [[400, 0], [0, 400]], [[7, 0], [0, 280]], [[288, 0], [0, 288]]]


@pytest.mark.parametrize("nload", [1, 3])
@pytest.mark.parametrize("M", PLANES, ids=[str(m) for m in PLANES])
def test_planes_match_oracle(fh, M, nload):
    case = Case(M, {"kind": "dlvp", "alpha": [0.25, 0.2]}, [(1.0, 0.3), (12.0, 0.2)], np.array([[0.1, -0.05]]), np.array([0.25]),
                nload=nload)
    s = case.product(fh)
    n = 6
    ref = case.oracle_solve(tol=0.0, max_iter=n)
    for prec, tol in ((fh.FH_PREC_FP64, 1e-10), (fh.FH_PREC_FP32, 5e-5)):
        out = s.solve(case.eps0, tol=0.0, max_iter=n, precision=prec, path=1)
        assert case.strain_error(s, ref["E"]) < tol, prec
        assert rel(out["mean_stress"], ref["mean_stress"]) < tol
    s.close()


@pytest.mark.parametrize("M", [[[20, 0], [0, 360]], [[18, 0], [0, 18]], [[2, 0, 0], [0, 36, 0], [0, 0, 36]], [[2, 0, 0], [0, 32, 0], [0, 0, 64]]],
                         ids=str)
def test_point_by_point_stiffness_matches_oracle(fh, M):
    """Every point its own matrix: the row pass reads the stiffness field (rows of
    32 and 64 points too, whose phase-wise solves take other passes)."""
    from oracle import green as OGr, material as OM, scheme as OS
    d = len(M)
    case = Case(M, {"kind": "dlvp", "alpha": [0.25] * d}, [(1.0, 0.3), (10.0, 0.3)], np.zeros((1, d)), np.array([0.3]), nload=2)
    y = case.T.points / case.T.D
    E = 1.0 + 9.0 * (0.5 + 0.5 * np.cos(2 * np.pi * y[:, -1])) + 0.01 * np.arange(len(y)) / len(y)
    lm = [OM.lame(e, 0.3) for e in E]
    C = np.stack([OM.isotropic_mandel(lam, mu, d) for lam, mu in lm])
    l0, m0 = OM.reference_medium_ms([q for q, _ in lm], [q for _, q in lm])
    C0 = OM.isotropic_mandel(l0, m0, d)
    Gp = OGr.gamma_p_table(case.M, case.gen_o, C0, case.T.freqs)
    s = case.product(fh)
    s.set_stiffness_field(np.ascontiguousarray(C[case.perm]))
    s.set_reference(None)
    for form in (0, 1):
        if form == 0:
            ref = OS.solve(case.T, Gp, C, C0, case.eps0, tol=0.0, max_iter=5)
        else:
            ref = OS.solve(case.T, Gp, C, C0, case.eps0, tol=0.0, max_iter=5, form="B")
        for prec, tol in ((fh.FH_PREC_FP64, 1e-10), (fh.FH_PREC_FP32, 5e-5)):
            s.solve(case.eps0, tol=0.0, max_iter=5, precision=prec, form=form)
            assert case.strain_error(s, ref["E"]) < tol, (form, prec)
    s.close()


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
