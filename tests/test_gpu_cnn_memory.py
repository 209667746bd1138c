"""Where a forward pass of the network may write, and how large it may be."""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def _net(seed=4):
    from paper_1609_00724_gb300 import qsl
    rng = np.random.default_rng(seed)
    d = ocnn.unflatten(ocnn.init_params(seed))
    d["b1"], d["b2"] = rng.uniform(-0.1, 0.1, 32), rng.uniform(-0.1, 0.1, 32)
    return qsl, qsl.Cnn(ocnn.flatten(d).astype(np.float32))


@pytest.mark.parametrize("n,h,w,at", [(1, 5, 7, 0), (6, 300, 260, 0), (6, 300, 260, 6 * 300 * 260), (3, 200, 130, 1001)])
def test_output_over_the_input(n, h, w, at):
    """prob in the memory of x (from its float `at` on): the same bits as beside it."""
    _, net = _net()
    x = torch.as_tensor(np.random.default_rng(n + at).normal(size=n * 2 * h * w).astype(np.float32)).cuda()
    want = net.forward(x.clone().view(n, 2, h, w))
    got = net.forward(x.view(n, 2, h, w), x[at:at + n * h * w].view(n, h, w))
    assert torch.equal(got, want)


@pytest.mark.parametrize("h,w", [(1, 2**31 - 1), (2**31 - 1, 1), (1, 2**31 - 2**22), (2**31 - 2**22, 1), (2**16, 2**16)])
def test_sides_beyond_32_bit_coordinates_are_refused(h, w):
    """Refused before anything is launched (the buffers here are small)."""
    qsl, net = _net()
    x = torch.zeros(64, device="cuda")
    L = qsl.lib()
    assert L.qsl_cnn_forward(net.handle, x.data_ptr(), 1, h, w, x.data_ptr(), None) == qsl.QSL_EINVAL
    assert b"CNN forward" in L.qsl_last_error()
