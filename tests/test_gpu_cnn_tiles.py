"""The tensor-core network kernels at the edges of their segments and tiles
(26, 58 or 122 columns forward, 30 x 12 data gradient, strips of at most 62
columns for the weight gradients) against the FP64 oracle, and with an infinite input."""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def _problem(seed, n, h, w):
    rng = np.random.default_rng(seed)
    d = ocnn.unflatten(ocnn.init_params(seed))
    d["b1"] = rng.uniform(-0.1, 0.1, 32)
    d["b2"] = rng.uniform(-0.1, 0.1, 32)
    d["b3"] = np.array([-0.2])
    x = rng.normal(size=(n, 2, h, w)).astype(np.float32)
    y = (rng.uniform(size=(n, h, w)) > 0.7).astype(np.float32)
    return ocnn.flatten(d).astype(np.float32), x, y


@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (3, 2, 1), (2, 1, 130), (1, 10, 26), (2, 11, 27), (1, 12, 30), (1, 13, 31),
                                   (2, 3, 62), (1, 5, 63), (1, 131, 3), (700, 3, 5), (1, 9, 58), (5, 7, 59), (1, 4, 122), (3, 2, 123)])
def test_tile_edges_match_oracle(n, h, w):
    """FP32 sums of at most 288 terms per output and n h w terms per gradient
    entry: 1e-5 of a probability, 1e-4 of a block's largest gradient, the
    bounds of the other network tests."""
    from paper_1609_00724_gb300 import qsl
    params, x, y = _problem(100 * h + w, n, h, w)
    net = qsl.Cnn(params)
    xd, yd = torch.as_tensor(x).cuda(), torch.as_tensor(y).cuda()
    z, _ = ocnn.forward(params.astype(np.float64), x.astype(np.float64))
    assert np.abs(net.forward(xd).cpu().numpy() - 1 / (1 + np.exp(-z))).max() < 1e-5
    loss, grad = torch.zeros(1, device="cuda"), torch.zeros(qsl.QSL_CNN_NPARAMS, device="cuda")
    net.loss_grad(xd, yd, 3.0, loss, grad)
    L, g = ocnn.loss_grad(params.astype(np.float64), x.astype(np.float64), y.astype(np.float64), 3.0)
    assert abs(loss.item() / L - 1) < 1e-5
    got, o = grad.cpu().numpy().astype(np.float64), 0
    for name, shp in ocnn.SHAPES:
        k = int(np.prod(shp))
        assert np.abs(got[o:o + k] - g[o:o + k]).max() <= 1e-4 * np.abs(g[o:o + k]).max() + 1e-9, name
        o += k


def test_infinite_input_stays_local():
    """An infinite pixel changes the 7 x 7 outputs that read it and no others."""
    from paper_1609_00724_gb300 import qsl
    params, x, _ = _problem(9, 1, 40, 70)
    net = qsl.Cnn(params)
    a = net.forward(torch.as_tensor(x).cuda()).cpu().numpy()
    x[0, 1, 20, 33] = np.inf
    b = net.forward(torch.as_tensor(x).cuda()).cpu().numpy()
    far = np.ones((40, 70), bool)
    far[17:24, 30:37] = False
    assert np.array_equal(a[0][far], b[0][far])
