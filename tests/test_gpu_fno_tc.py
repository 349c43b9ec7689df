"""The tensor-core row kernels against the SIMT ones at the edges of their range:
rows of 16 to 128 points, spectral rows that fill no group of 16, modes up to half
the axis, several samples, one to three layers (forward, gelu' and plain backward
forms).

Bounds: an output is a sum of at most 32 + 128 FP32 terms a layer, each operand
split to 2^-24, so two evaluations of up to three layers differ by at most about
3 x 160 x 2^-24 = 3e-5 of the largest partial sum, and by its square root's share
(2e-6) in the mean: 1e-5 of the largest output, 2e-5 in the norm of a gradient."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# n, modes, layers, batch
SIZES = [(16, 3, 2, 1), (16, 8, 3, 3), (32, 5, 2, 2), (48, 12, 2, 1), (64, 12, 2, 2), (128, 4, 1, 1), (128, 20, 2, 1)]


@pytest.mark.parametrize("size", SIZES, ids=["-".join(map(str, s)) for s in SIZES])
def test_tensor_cores_match_simt(size):
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    n, modes, layers, batch = size
    rng = np.random.default_rng(3)
    net = fh.FNO(n, 2, 5, 32, modes, layers, max_batch=batch)
    net.set_params((0.15 * rng.standard_normal(net.nparam)).astype(np.float32))
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(batch, 2, n ** 3, generator=g, device="cuda")
    t = torch.randn(batch, 5, n ** 3, generator=g, device="cuda")
    out = []
    for tc in (True, False):
        net.set_tensor_cores(tc)
        y = torch.empty(batch, 5, n ** 3, device="cuda")
        net.forward(x, y)
        net.zero_grad()
        loss = net.loss_grad(x, t)
        out.append((y.double(), loss, net.get_grads().astype(np.float64)))
    (ya, la, ga), (yb, lb, gb) = out
    assert float((ya - yb).abs().max() / yb.abs().max()) < 1e-5
    assert abs(la - lb) / lb < 1e-5
    W, nm = 32, 4 * modes ** 3
    o = 0
    for k in (2 * W, W, layers * W * W, layers * W, layers * nm * W * W, layers * nm * W * W, 5 * W, 5):
        a, b = ga[o:o + k], gb[o:o + k]
        assert np.linalg.norm(a - b) < 2e-5 * np.linalg.norm(b)
        o += k
    net.close()
