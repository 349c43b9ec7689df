"""Plates with two long axes (3-D, n_v = 6) on the FP32 passes: lengths whose column tile
holds eight columns and four, radices above 16 on rows and columns, each solved twice by
one solver so that the second solve replays the graph of the first.  Two plates against
the FP64 oracle, the larger ones against the solver's own FP64 passes, which take the
Stockham block passes at these lengths (above 256 points) and which the oracle pins in
the other parity tests.  Fixed point, mixed and BiCGStab; bounds of the other parity
tests."""
import numpy as np
import pytest

from parity import Case, rel

pytestmark = pytest.mark.gpu

ORACLE = [[2, 288, 288], [1, 576, 576]]
FP64 = [[2, 360, 360], [2, 480, 480], [2, 512, 512], [2, 576, 576], [2, 640, 640], [1, 768, 768], [2, 768, 768], [1, 1024, 1024],
        [8, 24, 576]]
N_IT = 4


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


def ids(d):
    return "x".join(map(str, d))


@pytest.mark.parametrize("dims", ORACLE, ids=ids)
def test_plates_match_oracle_twice(fh, dims):
    case = Case([[dims[0], 0, 0], [0, dims[1], 0], [0, 0, dims[2]]], {"kind": "dlvp", "alpha": [0.25, 0.2, 0.1]},
                [(1.0, 0.3), (12.0, 0.2)], np.array([[0.1, -0.05, 0.2]]), np.array([0.3]), nload=1)
    s = case.product(fh)
    ref = case.oracle_solve(tol=0.0, max_iter=N_IT)
    for prec, tol in ((fh.FH_PREC_FP32, 5e-5), (fh.FH_PREC_FP64, 1e-10)):
        for _ in range(2):   # chunk = max_iter: a whole replay
            out = s.solve(case.eps0, tol=0.0, max_iter=N_IT, precision=prec, chunk=N_IT, path=1)
            assert case.strain_error(s, ref["E"]) < tol, prec
            assert rel(out["mean_stress"], ref["mean_stress"]) < tol
    ref1 = case.oracle_solve(tol=0.0, max_iter=N_IT + 1)   # mixed: one more in FP64
    for _ in range(2):
        s.solve(case.eps0, tol=0.0, max_iter=N_IT, precision=fh.FH_PREC_MIXED, chunk=N_IT, path=1)
        assert case.strain_error(s, ref1["E"]) < 5e-5
    s.close()


@pytest.mark.parametrize("dims", FP64, ids=ids)
def test_plates_match_fp64_passes_twice(fh, dims):
    p = fh.Pattern([[dims[0], 0, 0], [0, dims[1], 0], [0, 0, dims[2]]])
    assert p.dims == [n for n in dims if n > 1]
    s = fh.Solver(p, fh.generator("dlvp", alpha=[0.25, 0.2, 0.1]), 2)
    ids = (np.random.default_rng(3).random(p.m) < 0.2).astype(np.uint8)
    s.set_stiffness_phases(ids, np.stack([fh.isotropic_stiffness(*fh.lame(E, nu), 3) for E, nu in ((1.0, 0.3), (12.0, 0.2))]))
    s.set_reference(None)
    eps0 = np.eye(6)[[0, 4]]

    def run(prec, method, n):
        out = s.solve(eps0, tol=0.0, max_iter=n, precision=prec, chunk=n, path=1, method=method)
        return np.stack([s.get_strain(k) for k in range(2)]), out["mean_stress"]

    for method, n in ((0, N_IT), (1, 2)):
        E64, m64 = run(fh.FH_PREC_FP64, method, n)
        scale = np.abs(E64 + eps0[:, :, None]).max()
        for _ in range(2):
            E, m = run(fh.FH_PREC_FP32, method, n)
            assert np.abs(E - E64).max() < 5e-5 * scale, method
            assert rel(m, m64) < 5e-5
    s.close()
