"""Waits of the network kernels that run out (qsl_check_cnn_waits gives the named
kernels no time at all): the launch ends, what depends on the kernel is NaN and
the rest as in an ordinary pass, and the network works as before afterwards.
Nothing waits on anything that does not come: MMAs under way are waited for
before their memory is freed."""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu

LAYERS = [name for name, _ in ocnn.SHAPES]


def _blocks(grad):
    got, o, out = grad.cpu().numpy(), 0, {}
    for name, shp in ocnn.SHAPES:
        k = int(np.prod(shp))
        out[name] = got[o:o + k]
        o += k
    return out


@pytest.fixture(scope="module")
def setup():
    """480 tiles of the data gradients and 288 of the weight gradients: more than
    one per block; an earlier pass on other data leaves its gradients in the
    buffers."""
    from paper_1609_00724_gb300 import qsl
    rng = np.random.default_rng(3)
    d = ocnn.unflatten(ocnn.init_params(3))
    d["b1"], d["b2"] = rng.uniform(-0.1, 0.1, 32), rng.uniform(-0.1, 0.1, 32)
    net = qsl.Cnn(ocnn.flatten(d).astype(np.float32))
    shape = (16, 64, 128)
    x, other = (torch.as_tensor(rng.normal(size=(16, 2, 64, 128)).astype(np.float32)).cuda() for _ in range(2))
    y = torch.as_tensor((rng.uniform(size=shape) > 0.7).astype(np.float32)).cuda()
    loss, grad = torch.zeros(1, device="cuda"), torch.zeros(qsl.QSL_CNN_NPARAMS, device="cuda")
    prob = net.forward(x)
    net.loss_grad(x, y, 1.0, loss, grad)
    want = prob.cpu().numpy(), loss.item(), _blocks(grad)
    return qsl, net, x, other, y, want


def _check(got, want, bad):
    for name in LAYERS:
        if name in bad:
            assert np.all(np.isnan(got[name])), name
        else:  # the order of the blocks' sums changes: FP32 rounding of at most some hundred terms
            assert np.abs(got[name] - want[name]).max() <= 1e-5 * np.abs(want[name]).max(), name


@pytest.mark.parametrize("kernels,bad", [(1, ()), (4, ("w2", "b2")), (8, ("w1", "b1", "w3")),
                                         (13, ("w1", "b1", "w2", "b2", "w3")), (0, ())])
def test_waits_that_run_out(setup, kernels, bad):
    qsl, net, x, other, y, (prob0, loss0, grad0) = setup
    prob, loss = torch.zeros_like(y), torch.zeros(1, device="cuda")
    grad = torch.zeros(qsl.QSL_CNN_NPARAMS, device="cuda")
    net.loss_grad(other, y, 1.0, loss, grad)
    net.check_waits(x, y, prob, loss, grad, kernels)
    got = prob.cpu().numpy()
    assert np.all(np.isnan(got)) if kernels & qsl.QSL_CNN_FORWARD else np.array_equal(got, prob0)
    assert abs(loss.item() / loss0 - 1) < 1e-5
    _check(_blocks(grad), grad0, bad)
    assert np.array_equal(net.forward(x).cpu().numpy(), prob0)
    net.loss_grad(x, y, 1.0, loss, grad)
    _check(_blocks(grad), grad0, ())


def test_missing_data_gradients_reach_both_layers(setup):
    """The data gradients' kernel stops at its first tile: layer 2's gradients,
    formed from buffers that still hold an earlier pass's values, are NaN like
    layer 1's."""
    qsl, net, x, other, y, (_, _, grad0) = setup
    prob, loss = torch.zeros_like(y), torch.zeros(1, device="cuda")
    grad = torch.zeros(qsl.QSL_CNN_NPARAMS, device="cuda")
    net.loss_grad(other, y, 1.0, loss, grad)
    net.check_waits(x, y, prob, loss, grad, qsl.QSL_CNN_DGRAD)
    _check(_blocks(grad), grad0, ("w1", "b1", "w2", "b2"))
