"""The loss of loss_grad over the range of its errors: squares beyond and below FP32's
range, infinities and NaN.  With all parameters zero the output is zero and the loss the
mean of target^2, which numpy gives in FP64; bound 4e-12 (32 squares a float pair, 2 x 32
roundings of 2^-24 of a part that is at most 32 x 2^-24 of the sum; the sums of the pairs
are FP64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fh():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    return fh


@pytest.mark.parametrize("n,cout", [(16, 36), (9, 5)])
def test_loss_over_the_range_of_its_errors(fh, n, cout):
    import torch
    net = fh.FNO(n, 1, cout, 8, 2, 1, max_batch=2)
    net.set_params(np.zeros(net.nparam, dtype=np.float32))
    rng = np.random.default_rng(11)
    x = torch.from_numpy(rng.standard_normal((2, 1, n ** 3)).astype(np.float32)).cuda()
    t0 = rng.standard_normal((2, cout, n ** 3))
    spread = 10.0 ** rng.uniform(-30, 30, t0.shape)
    for scale in (1.0, 1e30, 1e-25, 3e-17, 2e18, spread):
        t = (t0 * scale).astype(np.float32)
        net.zero_grad()
        loss = net.loss_grad(x, torch.from_numpy(t).cuda())
        ref = np.mean(t.astype(np.float64) ** 2)
        assert abs(loss - ref) <= 4e-12 * ref
    for special, want in ((np.inf, np.isposinf), (-np.inf, np.isposinf), (np.nan, np.isnan)):
        t = t0.astype(np.float32)
        t[1, cout // 2, 7] = special
        net.zero_grad()
        assert want(net.loss_grad(x, torch.from_numpy(t).cuda()))
    net.close()
