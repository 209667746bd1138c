"""The FP64 cell-wise tracer with sixteen lanes per line (line_lanes = 3 with
QSL_FP64, and the retrace of lines above retrace_q) against the one-lane FP64
kernel: one line, a handful, one line per warp, two lines per warp; both
interpolation modes; domains whose faces cut cells; a length cap."""
import numpy as np
import pytest

from paper_1609_00724_gb300 import inputs
from gpu_helpers import compare_lines

pytestmark = pytest.mark.gpu

# each kernel at tol 1e-10 is within 2e-6 (Q) and 3e-7 (float32 lengths) of the
# oracle (test_fp64_precision_matches_oracle_tightly); two of them, twice that
Q_RTOL2, L_RTOL2 = 4e-6, 6e-7


@pytest.fixture(scope="module")
def qsl():
    from paper_1609_00724_gb300 import qsl as q
    q.lib()
    return q


def _dict(rec):
    return {"q_perp": rec["q_perp"], "q_foot": rec["q_foot"], "q_det": rec["q_det"], "L": rec["length"],
            "face_f": rec["face_f"], "face_b": rec["face_b"], "xf": rec["x_f"], "xb": rec["x_b"],
            "st_f": rec["status_f"], "st_b": rec["status_b"]}


@pytest.mark.parametrize("count,mode,box,max_length",
                         [(1, 0, None, 0), (33, 1, None, 0), (700, 0, None, 0), (700, 1, "cut", 0), (3100, 0, "cut", 0),
                          (3100, 1, None, 0), (500, 0, None, 0.37)])
def test_sixteen_lanes_match_one_lane(qsl, count, mode, box, max_length):
    n = 29
    gf = inputs.charge_field(inputs.random_charges(4, 5), n)
    F = qsl.qsl_load_field(*(a.double().numpy() for a in (gf.bx, gf.by, gf.bz)), gf.xc, gf.yc, gf.zc, mode)
    seeds = inputs.random_seeds(count, 23 + count)
    lo, hi = np.array([-1.0, -1.0, 0.0]), np.array([1.0, 1.0, 1.0])
    kw = {}
    if box:
        lo, hi = np.array([-0.83, -1.0, 0.013]), np.array([0.91, 0.77, 0.98])
        seeds = np.clip(seeds, lo, hi)  # some on the cut faces
        kw = {"domain_lo": lo, "domain_hi": hi}
    rec = [qsl.qsl_trace_seeds(F, seeds, qsl.qsl_opts_default(
        tol_abs=1e-10, tol_rel=1e-10, precision=qsl.QSL_FP64, integrator=qsl.QSL_DOPRI5_CELL, line_lanes=lanes,
        max_length=max_length, **kw)) for lanes in (1, 3)]
    assert np.array_equal(rec[0]["status_f"], rec[1]["status_f"])
    assert np.array_equal(rec[0]["status_b"], rec[1]["status_b"])
    compare_lines(_dict(rec[1]), _dict(rec[0]), 1.0 / (n - 1), lo, hi, q_rtol=Q_RTOL2, l_rtol=L_RTOL2)
