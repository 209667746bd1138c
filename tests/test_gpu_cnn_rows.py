"""The network's forward pass where its blocks march through tall tasks and take
several groups of them, with an odd number of rows per group (the buffers' parity
flips between groups) and a last task that hangs over the image: one, two and
four segments per row step, against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


def _grid(n, H, W, slots):
    """Segment width, rows per task, overhang and groups of tasks that the launch
    takes for `slots` resident blocks."""
    P, tx = min(((P, -(-W // (P - 6))) for P in (32, 64, 128)), key=lambda c: c[0] * c[1])
    nseg = 128 // P
    groups = lambda ty: -(-n * tx * ty // nseg)
    ty = min(range(1, min(H, 1024) + 1), key=lambda ty: -(-groups(ty) // slots) * (-(-H // ty) + 4))
    h = -(-H // ty)
    ty = -(-H // h)
    return P, h, ty * h - H, groups(ty)


@pytest.mark.parametrize("n,h,w,segment", [(317, 19, 27, 32), (317, 19, 58, 64), (156, 19, 122, 128), (333, 61, 26, 32)])
def test_rows_and_groups_match_oracle(n, h, w, segment):
    """1e-5 of a probability, the bound of the other network tests."""
    from paper_1609_00724_gb300 import qsl
    slots = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    P, rows, hang, groups = _grid(n, h, w, slots)
    assert P == segment and rows >= 7 and (rows + 4) % 2 == 1 and hang > 0
    assert groups > slots or rows > 20
    rng = np.random.default_rng(w)
    d = ocnn.unflatten(ocnn.init_params(w))
    d["b1"], d["b2"], d["b3"] = rng.uniform(-0.1, 0.1, 32), rng.uniform(-0.1, 0.1, 32), np.array([-0.2])
    params = ocnn.flatten(d).astype(np.float32)
    x = rng.normal(size=(n, 2, h, w)).astype(np.float32)
    net = qsl.Cnn(params)
    xd = torch.as_tensor(x).cuda()
    got = net.forward(xd)
    assert torch.equal(got, net.forward(xd))
    worst = 0.0
    for i in range(0, n, 64):
        z, _ = ocnn.forward(params.astype(np.float64), x[i:i + 64].astype(np.float64))
        worst = max(worst, np.abs(got[i:i + 64].cpu().numpy() - 1 / (1 + np.exp(-z))).max())
    assert worst < 1e-5
