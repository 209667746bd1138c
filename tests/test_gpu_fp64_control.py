"""The step controller of the FP64 cell-wise tracers works in FP64 and in its
range, with one lane per line and with sixteen."""
import numpy as np
import pytest

from paper_1609_00724_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qsl():
    from paper_1609_00724_gb300 import qsl as q
    q.lib()
    return q


def _opts(qsl, lanes, **kw):
    return qsl.qsl_opts_default(tol_abs=1e-10, tol_rel=1e-10, precision=qsl.QSL_FP64, integrator=qsl.QSL_DOPRI5_CELL,
                                line_lanes=lanes, **kw)


@pytest.mark.parametrize("lanes", [1, 3])
def test_first_step_of_any_size(qsl, lanes):
    """A first step far below FP32's range grows by 5 per step and gives the
    lines of the default one: each within 2e-6 (Q) and 3e-7 (length) of the
    oracle at this tolerance, two of them twice that."""
    gf = inputs.charge_field(inputs.random_charges(4, 5), 29)
    F = qsl.qsl_load_field(*(a.double().numpy() for a in (gf.bx, gf.by, gf.bz)), gf.xc, gf.yc, gf.zc, 0)
    seeds = inputs.random_seeds(60, 3)
    a, b = [qsl.qsl_trace_seeds(F, seeds, _opts(qsl, lanes, h_init=h, max_steps=4000)) for h in (0.1, 1e-60)]
    for k in ("face_f", "face_b", "status_f", "status_b"):
        assert np.array_equal(a[k], b[k]), k
    assert np.allclose(a["q_perp"], b["q_perp"], rtol=4e-6, atol=0, equal_nan=True)
    assert np.allclose(a["length"], b["length"], rtol=6e-7, atol=0)


@pytest.mark.parametrize("lanes", [1, 3])
def test_deviations_beyond_fp32_range(qsl, lanes):
    """The axis of B = (lam x, -lam y, b0): deviations grow by e^(lam / b0) = 1e52
    and the error of a step relative to them stays what the tolerance asks, so
    Q = k^2 + 1 / k^2 with k = e^(lam / b0) is met to a step count of at most
    some thousand times the tolerance (1e-10), twice."""
    lam = 120.0
    gf = inputs.hyperbolic_field(17, lam, 1.0)
    F = qsl.qsl_load_field(gf.bx, gf.by, gf.bz, gf.xc, gf.yc, gf.zc, qsl.QSL_RAW_B)
    rec = qsl.qsl_trace_seeds(F, np.array([[0.0, 0.0, 0.0]]), _opts(qsl, lanes))
    assert rec["face_f"][0] == 5 and rec["status_f"][0] == qsl.QSL_LINE_OK
    k2 = np.exp(2 * lam)
    assert abs(rec["q_foot"][0] / k2 - 1) < 1e-6, (rec["q_foot"][0], k2)
