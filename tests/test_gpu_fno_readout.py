"""Parameters and gradients read out with no room left on the device for the buffer that
takes the complex weights apart: the same numbers as with it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_read_out_without_device_memory():
    import torch
    assert torch.cuda.is_available()
    from paper_1701_04685_gb300 import build
    build.build()
    import paper_1701_04685_gb300 as fh
    nets, sets = [], []
    for full in (False, True):
        net = fh.FNO(24, 1, 6, 32, 12, 4, max_batch=1)   # 57 M parameters
        g = torch.Generator(device="cuda").manual_seed(5)
        prm = (0.1 * torch.randn(net.nparam, generator=g, device="cuda")).cpu().numpy()
        net.set_params(prm)
        x = torch.randn(1, 1, 24 ** 3, generator=g, device="cuda")
        t = torch.randn(1, 6, 24 ** 3, generator=g, device="cuda")
        net.zero_grad()
        net.loss_grad(x, t)
        fill = None
        if full:
            torch.cuda.empty_cache()
            room = net.nparam * 4 // 2
            fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        sets.append((prm, net.get_params(), net.get_grads()))
        del fill
        torch.cuda.empty_cache()
        nets.append(net)
    for prm, got, _ in sets:
        assert np.array_equal(prm, got)
    # gradients: sums of the weights' blocks differ in order between two runs
    a, b = sets[0][2], sets[1][2]
    assert np.abs(a).max() > 0 and np.abs(a - b).max() <= 1e-5 * np.abs(a).max()
    for net in nets:
        net.close()
