"""Network features of slices on either side of the rule that gives a slice one
block or a cluster of eight, against plain FP64: the slice's largest finite value
anywhere in it, missing and infinite entries."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,ny,nx", [(1, 1, 1), (1, 32, 32), (1, 5, 205), (600, 8, 8), (26, 33, 31), (25, 32, 33),
                                      (410, 128, 128), (409, 128, 128), (410, 127, 129), (2, 300, 200)])
def test_features_match_fp64(nz, ny, nx):
    from paper_1609_00724_gb300 import qsl
    rng = np.random.default_rng(nz + ny)
    S = rng.exponential(size=(nz, ny, nx)).astype(np.float32)
    Q = (2 + 10 ** rng.uniform(-1, 9, size=S.shape)).astype(np.float32)
    at = rng.integers(0, ny * nx, nz)
    S.reshape(nz, -1)[np.arange(nz), at] = 50.0 + np.arange(nz)
    for v in (np.nan, np.inf, -np.inf):
        S[rng.uniform(size=S.shape) < 0.01] = v
        Q[rng.uniform(size=S.shape) < 0.01] = v
    s, q, X = torch.as_tensor(S).cuda(), torch.as_tensor(Q).cuda(), torch.empty((nz, 2, ny, nx), device="cuda")
    assert qsl.lib().qsl_cnn_features(s.data_ptr(), q.data_ptr(), nz, ny, nx, X.data_ptr(), None) == qsl.QSL_OK
    X = X.cpu().numpy()
    fin = np.where(np.isfinite(S), S, 0).astype(np.float64)
    want = fin / np.maximum(fin.reshape(nz, -1).max(1), 1e-12).reshape(-1, 1, 1)
    # one FP32 division; log10f within 2 ulp of values up to 9, halved
    assert np.abs(X[:, 0] - want).max() <= 2.0**-24 * 2
    q64 = np.where(np.isnan(Q) | (Q == -np.inf), 2.0, Q.astype(np.float64))
    want = np.where(np.isinf(q64), 3.0, np.clip((np.log10(np.maximum(q64, 2.0)) - 2) * 0.5, -2, 3))
    assert np.abs(X[:, 1] - want).max() <= 1.5e-6
