"""Weight gradients of networks with at most eight channels on either side, whose tiles have
eight rows or columns, and around that line: against the FP64 oracle's central finite
differences along a random direction of each parameter block, within 2e-3 (the bound of
the other network tests).  Voxel counts that are and are not multiples of four."""
import numpy as np
import pytest

from oracle import fno as OF
from test_gpu_fno import bf16

pytestmark = pytest.mark.gpu

# n, cin, cout, width, modes, layers, batch
SIZES = [(8, 1, 36, 1, 2, 1, 2), (8, 8, 8, 8, 2, 1, 1), (6, 9, 9, 8, 2, 1, 2), (8, 7, 6, 9, 3, 1, 1), (5, 1, 40, 2, 2, 2, 3), (7, 33, 3, 3, 1, 1, 1)]


@pytest.mark.parametrize("size", SIZES, ids=["-".join(map(str, s)) for s in SIZES])
def test_weight_gradients(size):
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    n, cin, cout, width, modes, layers, batch = size
    rng = np.random.default_rng(17)
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
    net.zero_grad()
    net.loss_grad(torch.from_numpy(x.reshape(batch, cin, -1)).cuda(), torch.from_numpy(t.reshape(batch, cout, -1)).cuda())
    g = net.get_grads().astype(np.float64)
    xs, ts = list(x.astype(np.float64)), list(t.astype(np.float64))
    theta = p.flat()
    q = OF.Params(cin, cout, width, modes, layers)
    o = 0
    for name, k in zip(("P", "p", "W", "w", "ReR", "ImR", "Q", "q"),
                       (p.P.size, p.p.size, p.W.size, p.w.size, p.R.size, p.R.size, p.Q.size, p.q.size)):
        d = np.zeros_like(theta)
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
