"""Gamma^p tables for reference media that are not isotropic (and for box splines
whose directions are not unit vectors) against the FP64 oracle: orthotropic and
fully anisotropic C0, separable and non-separable symbols, diagonal patterns
(whose mirror images share one alias sum) of odd, even and unequal lengths, and
sheared ones.

Bound: the tables agree to 1e-12 relative to their largest entry (as the other
table tests): about 100 roundings of 1.1e-16 per alias term and the sum of at
most 7^3 aliases of one weight total.
"""
import numpy as np
import pytest

from oracle import generators as OG, green as OGr, scheme as OS
from parity import product_generator, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


def reference(kind, d):
    rng = np.random.default_rng(40 + d)
    n = 3 if d == 2 else 6
    A = rng.standard_normal((n, n))
    C = A @ A.T + n * np.eye(n)
    if kind == "orthotropic":
        C[:d, d:] = 0.0
        C[d:, :d] = 0.0
        C[d:, d:] = np.diag(np.diag(C)[d:])
    return C


GENS = {
    "dirichlet": lambda d: {"kind": "dirichlet"},
    "dlvp": lambda d: {"kind": "dlvp", "alpha": [0.25, 0.1, 0.4][:d]},
    "box": lambda d: {"kind": "boxspline", "order": 2, "radius": 2},
    "courant": lambda d: {"kind": "boxspline", "radius": 2,
                          "xi": np.concatenate([np.eye(d)] * 2 + [np.ones((d, 1))], axis=1)},
}
PATTERNS = [[[8, 0], [0, 8]], [[6, 2], [0, 9]], [[5, 0, 0], [0, 5, 0], [0, 0, 5]],
            [[4, 0, 0], [0, 4, 0], [0, 0, 8]], [[4, 0, 0], [0, 6, 0], [0, 0, 10]], [[4, 1, 0], [0, 5, 2], [0, 0, 6]]]


@pytest.mark.parametrize("kind", ["orthotropic", "anisotropic"])
@pytest.mark.parametrize("gen", list(GENS))
@pytest.mark.parametrize("M", PATTERNS, ids=[str(m) for m in PATTERNS])
def test_table_matches_oracle(fh, M, gen, kind):
    d = len(M)
    C0 = reference(kind, d)
    spec = GENS[gen](d)
    if spec["kind"] == "boxspline":
        xi = spec.get("xi", np.concatenate([np.eye(d)] * 2, axis=1))
        og = OG.Generator("boxspline", xi=np.asarray(xi, float), radius=spec["radius"])
    else:
        og = OG.Generator(**spec)
    T = OS.SNFTransform(M)
    p = fh.Pattern(M)
    s = fh.Solver(p, product_generator(fh, spec, d), 1)
    s.set_stiffness_phases(np.zeros(p.m, dtype=np.uint8), C0[None])
    s.set_reference(C0)
    ref = OGr.gamma_p_table(M, og, C0, p.half_freqs())
    assert T.D == p.m
    assert rel(s.get_green(), ref) < 1e-12
    s.close()
