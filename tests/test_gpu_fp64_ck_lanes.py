"""The FP64 Cash-Karp tracer with sixteen lanes per line (line_lanes = 0, few
lines, and the retrace of lines above retrace_q) against the one-lane kernel:
one line, one per warp, two per warp; both interpolation modes; domains whose
faces cut cells, seeds on faces and outside; a length cap; tight tolerances."""
import numpy as np
import pytest
import torch

from paper_1609_00724_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsl():
    from paper_1609_00724_gb300 import qsl as q
    q.lib()
    return q


def _field(qsl, n, mode, seed=5):
    gf = inputs.charge_field(inputs.random_charges(4, seed), n)
    return qsl.qsl_load_field(*(a.double().numpy() for a in (gf.bx, gf.by, gf.bz)), gf.xc, gf.yc, gf.zc, mode)


@pytest.mark.parametrize("count,mode,box,max_length,tol",
                         [(1, 0, None, 0, 1e-2), (33, 1, None, 0, 1e-2), (700, 0, None, 0, 1e-4), (700, 1, "cut", 0, 1e-2),
                          (3100, 0, "cut", 0, 1e-3), (12000, 1, None, 0, 1e-2), (500, 0, None, 0.37, 1e-3),
                          (300, 0, None, 0, 1e-6)])
def test_sixteen_lanes_match_one_lane(qsl, count, mode, box, max_length, tol):
    """Same method, steps and precision: FP64 rounding (1e-16) grown along lines
    of some hundred steps (some thousand at 1e-6), against 1e-8 (1e-4)."""
    F = _field(qsl, 29, mode)
    seeds = inputs.random_seeds(count, 23 + count)
    kw = {}
    if box:
        lo, hi = np.array([-0.83, -1.0, 0.013]), np.array([0.91, 0.77, 0.98])
        seeds[1::2] = np.clip(seeds[1::2], lo, hi)  # some on the cut faces, some outside
        kw = {"domain_lo": lo, "domain_hi": hi}
    a, b = [qsl.qsl_trace_seeds(F, seeds, qsl.qsl_opts_default(
        tol_abs=tol, tol_rel=tol, precision=qsl.QSL_FP64, integrator=qsl.QSL_RKCK54, line_lanes=lanes,
        max_length=max_length, **kw)) for lanes in (1, 0)]
    for k in ("face_f", "face_b", "status_f", "status_b"):
        assert np.array_equal(a[k], b[k]), k
    rtol = 1e-8 if tol > 1e-5 else 1e-4
    for k in ("q_perp", "q_foot", "q_det"):
        assert np.allclose(a[k], b[k], rtol=rtol, atol=0, equal_nan=True), k
    assert np.allclose(a["length"], b["length"], rtol=1e-6, atol=0, equal_nan=True)
    assert np.allclose(a["x_f"], b["x_f"], rtol=0, atol=2e-7, equal_nan=True) and np.allclose(a["x_b"], b["x_b"], rtol=0, atol=2e-7, equal_nan=True)


@pytest.mark.parametrize("retrace_q", [3.0, 200.0])
def test_retrace_list_on_either_side_of_the_rule(qsl, retrace_q):
    """The retrace list's length is known on the device only: a long list
    (one lane) and a short one (sixteen) replace the same lines."""
    F = _field(qsl, 33, 0)
    m = 300
    out = []
    for lanes in (1, 0):
        q, L = torch.empty(m * m, device="cuda"), torch.empty(m * m, device="cuda")
        o = qsl.qsl_opts_default(integrator=qsl.QSL_RKCK54, retrace_q=retrace_q, line_lanes=lanes)
        qsl.qsl_q_map_2d(F, (0, 0, 0), (2, 0, 0), (0, 2, 0), m, m, o, q=q, length=L)
        out.append((q.cpu().numpy(), L.cpu().numpy()))
    assert np.allclose(out[0][0], out[1][0], rtol=1e-6, atol=0, equal_nan=True)
    assert np.allclose(out[0][1], out[1][1], rtol=1e-6, atol=0, equal_nan=True)
