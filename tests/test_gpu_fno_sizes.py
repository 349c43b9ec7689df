"""The network's kernels at the edges of their tiles, against the FP64 network
oracle: rows that are no multiple of four points, channels that fill no group of
eight or 32, a single channel and mode, modes up to half the axis, batches that
straddle the voxel chunks of the weight gradient, several blocks of the mixing
matrices, an odd number of parameters before R.  Forward within 2e-5 of the largest value, the gradient along a random
direction of every parameter block within 2e-3 of the oracle's central finite
difference (the bounds of the other network tests)."""
import numpy as np
import pytest

from oracle import fno as OF
from test_gpu_fno import bf16

pytestmark = pytest.mark.gpu

# n, cin, cout, width, modes, layers, batch
SIZES = [(4, 1, 1, 1, 1, 1, 1), (5, 2, 3, 2, 2, 2, 3), (8, 7, 6, 33, 4, 1, 2), (15, 3, 5, 5, 7, 2, 2), (20, 1, 36, 12, 10, 1, 3),
         (22, 9, 41, 17, 5, 1, 2), (16, 1, 4, 56, 2, 1, 1), (40, 1, 2, 8, 3, 1, 1),
         (6, 2, 3, 5, 3, 1, 2)]


@pytest.mark.parametrize("size", SIZES, ids=["-".join(map(str, s)) for s in SIZES])
def test_forward_and_gradient_match_oracle(size):
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    n, cin, cout, width, modes, layers, batch = size
    rng = np.random.default_rng(7)
    p = OF.Params(cin, cout, width, modes, layers)
    p.P = rng.standard_normal(p.P.shape) / np.sqrt(cin)
    p.p = 0.1 * rng.standard_normal(p.p.shape)
    p.W = bf16(rng.standard_normal(p.W.shape) / np.sqrt(width))
    p.w = 0.1 * rng.standard_normal(p.w.shape)
    p.R = (bf16(rng.standard_normal(p.R.shape)) + 1j * bf16(rng.standard_normal(p.R.shape))) / 64.0
    p.Q = rng.standard_normal(p.Q.shape) / np.sqrt(width)
    p.q = 0.1 * rng.standard_normal(p.q.shape)
    p.set_flat(p.flat().astype(np.float32).astype(np.float64))
    net = fh.FNO(n, cin, cout, width, modes, layers, max_batch=batch)
    net.set_params(p.flat().astype(np.float32))
    x = rng.standard_normal((batch, cin, n, n, n)).astype(np.float32)
    t = rng.standard_normal((batch, cout, n, n, n)).astype(np.float32)
    xd = torch.from_numpy(x.reshape(batch, cin, -1)).cuda()
    y = torch.empty((batch, cout, n ** 3), dtype=torch.float32, device="cuda")
    net.forward(xd, y)
    got = y.cpu().numpy().reshape(batch, cout, n, n, n)
    xs, ts = list(x.astype(np.float64)), list(t.astype(np.float64))
    for b in range(batch):
        ref = OF.forward(p, xs[b])
        assert np.abs(got[b] - ref).max() / np.abs(ref).max() < 2e-5
    net.zero_grad()
    loss = net.loss_grad(xd, torch.from_numpy(t.reshape(batch, cout, -1)).cuda())
    ref_loss = OF.loss(p, xs, ts)
    assert abs(loss - ref_loss) / ref_loss < 1e-5
    g = net.get_grads().astype(np.float64)
    theta = p.flat()
    q = OF.Params(cin, cout, width, modes, layers)
    o = 0
    for name, k in zip(("P", "p", "W", "w", "ReR", "ImR", "Q", "q"),
                       (p.P.size, p.p.size, p.W.size, p.w.size, p.R.size, p.R.size, p.Q.size, p.q.size)):
        d = np.zeros_like(theta)
        # along the gradient's own sign, so that the derivative is not small against its terms
        d[o:o + k] = np.where(g[o:o + k] < 0, -1.0, 1.0) * rng.uniform(0.5, 1.0, k)
        h = 1e-4
        q.set_flat(theta + h * d)
        lp = OF.loss(q, xs, ts)
        q.set_flat(theta - h * d)
        lm = OF.loss(q, xs, ts)
        fd, an = (lp - lm) / (2 * h), float(g @ d)
        assert abs(fd - an) <= 2e-3 * abs(fd) + 1e-9, (name, fd, an)
        o += k
    net.close()
